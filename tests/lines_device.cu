// Interleaved FP64 lines of one CTA (csrc/cplx.cuh, CtaFft) whose scales differ by
// powers of two up to 2^-600, against long double sums: prints n, lines, direction and
// the largest relative L2 error of a line.
#include <cmath>
#include <complex>
#include <cstdio>
#include <vector>

#include "cplx.cuh"

using namespace tdse;
typedef std::complex<long double> cl;

template <int N, int L, int LS, int T, bool INV> __global__ void k_lines(double2* x, const int4* tw) {
    extern __shared__ __align__(16) unsigned char sm[];
    double2* buf = reinterpret_cast<double2*>(sm);
    for (int i = threadIdx.x; i < N * L; i += T) buf[(i / L) * LS + i % L] = x[i];
    __syncthreads();
    CtaFft<double2, N, L, LS, T, INV>::run(buf, tw, nullptr);
    for (int i = threadIdx.x; i < N * L; i += T) x[i] = buf[(i / L) * LS + i % L];
}

template <int N, int L, int LS, int T, bool INV> static int check() {
    std::vector<int4> tw(N);
    std::vector<cl> w(N);
    for (int m = 0; m < N; ++m) {
        const long double t = 2 * 3.141592653589793238462643383279502884L * m / N;
        fx_limbs(llroundl(cosl(t) * 0x1p61L), tw[m].x, tw[m].y);
        fx_limbs(llroundl(-sinl(t) * 0x1p61L), tw[m].z, tw[m].w);
        w[m] = cl(cosl(t), (INV ? 1 : -1) * sinl(t));
    }
    const int scale[8] = {0, -20, -300, -45, 3, -600, -56, -1};
    std::vector<double2> x(N * L), y(N * L);
    for (int i = 0; i < N * L; ++i)
        x[i] = make_double2(std::ldexp(std::sin(0.9 * i + 0.1 * i * i), scale[i % L]), std::ldexp(std::cos(1.7 * i * i), scale[i % L]));
    void *dx, *dt;
    const size_t smem = (size_t)N * LS * 16;
    if (cudaMalloc(&dx, x.size() * 16) != cudaSuccess || cudaMalloc(&dt, tw.size() * 16) != cudaSuccess) return 2;
    cudaMemcpy(dx, x.data(), x.size() * 16, cudaMemcpyHostToDevice);
    cudaMemcpy(dt, tw.data(), tw.size() * 16, cudaMemcpyHostToDevice);
    if (cudaFuncSetAttribute(k_lines<N, L, LS, T, INV>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return 2;
    k_lines<N, L, LS, T, INV><<<1, T, smem>>>((double2*)dx, (const int4*)dt);
    if (cudaGetLastError() != cudaSuccess || cudaMemcpy(y.data(), dx, y.size() * 16, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    cudaFree(dx);
    cudaFree(dt);
    long double worst = 0;
    for (int l = 0; l < L; ++l) {
        long double e = 0, n2 = 0;
        for (int k = 0; k < N; ++k) {
            cl s = 0;
            for (int j = 0; j < N; ++j) s += cl(x[j * L + l].x, x[j * L + l].y) * w[(long long)j * k % N];
            s *= powl(2.0L, -scale[l]);
            e += std::norm(cl(y[k * L + l].x, y[k * L + l].y) * powl(2.0L, -scale[l]) - s);
            n2 += std::norm(s);
        }
        worst = std::max(worst, sqrtl(e / n2));
    }
    std::printf("%d %d %d %.3Le\n", N, L, (int)INV, worst);
    return 0;
}

int main() {
    return check<8, 4, 4, 64, false>() || check<16, 4, 5, 64, true>() || check<64, 4, 4, 64, false>() || check<256, 4, 5, 128, true>() ||
           check<1024, 4, 4, 512, false>() || check<128, 8, 9, 256, true>() || check<512, 8, 8, 256, false>() ||
           check<128, 1, 1, 256, false>();
}
