// 1D periodic FP64 solves of n <= 1024: a whole run of time steps (start-up
// chains included) in one launch, one CTA per instance, one or two modes per
// thread.
//
// Bound by latency: a step is a chain of history sum -> inverse transform ->
// implicit solve -> forward transform -> update of a few thousand points, with
// nothing else for the SM to do when the batch is small.  So
//  * the mode state, the history and its phase factors stay in registers from
//    step to step (a step reads two phase factors and V, writes one ring slot);
//  * every thread owns one mode (two at n = 1024): the kernel this replaces gave
//    a thread eight and left n = 128 to 16 threads;
//  * the transforms are radix 4 (half the serial work of radix 8 per pass) in
//    64-bit fixed point (fx.cuh), ping-pong between two shared buffers, one
//    barrier per pass, and stay in fixed point across the implicit solve, whose
//    factor V / (1 + i beta) is formed per point beforehand.
// Against one launch per step of the kernel that larger n use, 100 steps:
// n = 128 x 1 9.1 -> 0.88 ms, 64 x 2048 25.1 -> 3.7, 512 x 1 10.0 -> 1.65,
// 512 x 400 14.0 -> 5.1, 1024 x 1 11.5 -> 3.2, 1024 x 200 18.4 -> 6.3.
#include "device_once.h"
#include "step_common.cuh"

namespace tdse {
namespace {

constexpr int RUN1D64_MAX = 1024;

template <int N> struct Run1D64 {
    static constexpr int T = N < 32 ? 32 : (N > 512 ? 512 : N);
    static constexpr int PER = N > T ? N / T : 1;
    static constexpr int LEN = N + N / 8;                    // padded: pos + pos / 8
    static constexpr size_t smem = (2 * (size_t)LEN + N) * 16;   // two transform buffers, the solve's factors
};
__device__ __forceinline__ int pad8(int p) { return p + (p >> 3); }

// Largest v over the CTA; slot: one of the reductions of a step (a slot is
// written again only after later barriers of the same step).
template <int T>
__device__ __forceinline__ unsigned cta_max(unsigned v, int slot) {
    __shared__ unsigned red[3][32];
    v = __reduce_max_sync(0xffffffffu, v);
    if constexpr (T > 32) {
        if ((threadIdx.x & 31) == 0) red[slot][threadIdx.x >> 5] = v;
        __syncthreads();
        v = __reduce_max_sync(0xffffffffu, red[slot][(threadIdx.x & 31) % (T / 32)]);
    }
    return v;
}

// Passes S.. of a transform of N points in X (results in the returned buffer),
// radix-4 butterflies by threads tid < N / R; the barrier before the first
// read is the caller's, each pass ends with one.
template <int N, bool INV, int S, int LAST>
__device__ __forceinline__ void passes(longlong2*& X, longlong2*& Y, const int4* __restrict__ tw) {
    using Plan = FftPlan4<N, INV>;
    using Fx = FxPass<N, INV, Plan>;
    using G = Run1D64<N>;
    if constexpr (S <= LAST) {
        constexpr int R = Plan::radix(S), Ns = Plan::ns(S), NB = N / R;
        static_assert(NB <= G::T, "one butterfly per thread");
        const int j = threadIdx.x;
        if (j < NB) {
            longlong2 v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = X[pad8(j + r * NB)];
            Fx::template butterfly<S>(v, j, tw);
            const int k = j & (Ns - 1), base = (j - k) * R + k;
#pragma unroll
            for (int r = 0; r < R; ++r) Y[pad8(base + r * Ns)] = v[r];
        }
        __syncthreads();
        longlong2* t = X;
        X = Y;
        Y = t;
        passes<N, INV, S + 1, LAST>(X, Y, tw);
    }
}

// R = DFT(V IDFT(W) / (1 + i hmu0 V)) / N of the CTA's instance: W and R in the
// registers of the mode owners, V of the same positions.
template <int N>
__device__ __forceinline__ void core(const double2 (&W)[Run1D64<N>::PER], const double (&V)[Run1D64<N>::PER],
                                     double hmu0, double2 (&R)[Run1D64<N>::PER], longlong2* A, longlong2* B, int4* Q,
                                     const int4* __restrict__ tw) {
    using G = Run1D64<N>;
    using PI = FftPlan4<N, true>;
    using PF = FftPlan4<N, false>;
    using FI = FxPass<N, true, PI>;
    using FF = FxPass<N, false, PF>;
    constexpr int RL = PI::radix(PI::NPASS - 1), NBL = N / RL;   // last inverse pass = first forward pass
    static_assert(RL == PF::radix(0), "the solve works on the last inverse butterfly's outputs");
    const int tid = threadIdx.x;
    double2 q[G::PER];
    unsigned mw = 0, mq = 0;
#pragma unroll
    for (int p = 0; p < G::PER; ++p) {
        const double beta = hmu0 * V[p], qx = V[p] * recip_ge1(fma(beta, beta, 1.0));
        q[p] = make_double2(qx, -beta * qx);
        if (N < G::T && tid + p * G::T >= N) continue;      // n = 8, 16: threads without a mode of their own
        mw = max(mw, fx_hi(W[p]));
        mq = max(mq, fx_hi(q[p]));
    }
    // one reduction for both (exponents: high 11 bits, the low bits do not matter)
    mw = cta_max<G::T>(mw, 0);
    mq = cta_max<G::T>(mq, 1);
    const int E = fx_exponent(mw), Eq = fx_exponent(mq);
    constexpr int SQ = 60;                       // |q| below 2^60.5: a factor of modulus below 0.71
#pragma unroll
    for (int p = 0; p < G::PER; ++p) {
        const int m = tid + p * G::T;
        if (N >= G::T || m < N) {
            A[pad8(m)] = fx_from(W[p], FI::S0, E);
            Q[m] = fx_as_factor(fx_from(q[p], SQ, Eq));
        }
    }
    __syncthreads();
    longlong2 *X = A, *Y = B;
    passes<N, true, 0, PI::NPASS - 2>(X, Y, tw);
    // last inverse pass, implicit solve and V u, first forward pass: in registers
    longlong2 v[RL];
    unsigned my = 0;
    if (tid < NBL) {
#pragma unroll
        for (int r = 0; r < RL; ++r) v[r] = X[pad8(tid + r * NBL)];
        if constexpr (PI::NPASS == 1) dft_r<RL, true>(v);
        else FI::template butterfly<PI::NPASS - 1>(v, tid, tw);
#pragma unroll
        for (int r = 0; r < RL; ++r) {
            const int hx = (int)(v[r].x >> 32), hy = (int)(v[r].y >> 32);
            my = max(my, max((unsigned)(hx ^ (hx >> 31)), (unsigned)(hy ^ (hy >> 31))));
        }
    }
    my = cta_max<G::T>(my, 2);                   // y fills its 62 bits before the forward transform scales it down
    const int sft = max(__clz((int)my) - 2, 0);
    constexpr int K = 3 - ilog2(RL);             // the product leaves room for the first forward butterfly
    if (tid < NBL) {
#pragma unroll
        for (int r = 0; r < RL; ++r) {
            v[r] = make_longlong2((long long)((unsigned long long)v[r].x << sft), (long long)((unsigned long long)v[r].y << sft));
            v[r] = fx_mul<false, K>(v[r], Q[tid + r * NBL]);
        }
        dft_r<RL, false>(v);
#pragma unroll
        for (int r = 0; r < RL; ++r) Y[pad8(tid * RL + r)] = v[r];
    }
    __syncthreads();
    longlong2* t = X;
    X = Y;
    Y = t;
    passes<N, false, 1, PF::NPASS - 1>(X, Y, tw);
    const bool bad = max(mw, mq) >= 0x7ff00000u;
    const int xy = E - 1022 - FI::S0 + FI::GAIN - sft;                 // y = v 2^xy
    const int xr = xy + Eq - 1022 - SQ + 64 - K + FF::GAIN - ilog2(N);
#pragma unroll
    for (int p = 0; p < G::PER; ++p) {
        const int m = tid + p * G::T;
        R[p] = (N >= G::T || m < N) ? fx_to(X[pad8(m)], bad ? FX_NAN : xr) : make_double2(0.0, 0.0);
    }
    __syncthreads();                             // the buffers are free again
}

template <int N>
__global__ void __launch_bounds__(Run1D64<N>::T, 1) k_run1d64(const __grid_constant__ KArgs a,
                                                           const __grid_constant__ Run1DArgs g) {
    using G = Run1D64<N>;
    constexpr int PER = G::PER, T = G::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    longlong2* A = reinterpret_cast<longlong2*>(smem_raw);
    longlong2* B = A + G::LEN;
    int4* Q = reinterpret_cast<int4*>(B + G::LEN);
    const int b = blockIdx.x, tid = threadIdx.x;
    double2* st = reinterpret_cast<double2*>(a.uhat) + (size_t)b * N;
    double2* ring = reinterpret_cast<double2*>(a.ring) + (size_t)b * a.ring_slots * N;
    const double* tfac = a.tfac + (size_t)b * a.ntf;
    const double* V0 = a.V0 + (size_t)b * a.vstride;
    const int4* adv = a.adv64 + (size_t)b * a.n_int * (size_t)(a.nh + a.nl);
    const int4* tw = a.tw64_0;
    const int RS = a.ring_slots;
    int mode[PER];
#pragma unroll
    for (int p = 0; p < PER; ++p) mode[p] = N >= T ? tid + p * T : (tid < N ? tid : N - 1);
    const bool own = N >= T || tid < N;

    auto main_iv = [&](int n) {
        return n <= g.S_eff ? (n - 1) * ((1 << g.L) - 1) : g.n_int_startup + (n - g.S_eff - 1);
    };
    // one-step phase factor over interval iv with the kinetic part of step size dt / 2^kin
    auto factor = [&](int iv, int kin, int m) {
        const int4* t = adv + (size_t)iv * (size_t)(a.nh + a.nl);
        const int4 w = fx_as_factor(fx_mul<false, 3>(fx_value(__ldg(&t[m >> a.lb])), __ldg(&t[a.nh + (m & (a.nl - 1))])));
        return fx_as_factor(fx_mul<false, 3>(fx_value(__ldg(&a.kin64[(size_t)kin * N + m])), w));
    };
    double V0r[PER];
#pragma unroll
    for (int p = 0; p < PER; ++p) V0r[p] = g.vtable ? 0.0 : V0[mode[p]];
    auto potential = [&](int tf, double (&V)[PER]) {
        const double f = tfac[tf];
        const int fine = 8 * g.S_eff;
        const size_t row = (size_t)(tf <= fine ? tf : fine + (tf / 8 - g.S_eff)) * N;
#pragma unroll
        for (int p = 0; p < PER; ++p) V[p] = f * (g.vtable ? V0[row + mode[p]] : V0r[p]);
    };

    double2 u[PER], r[PER][MAX_HIST], W[PER], R[PER];
    int4 w[PER][MAX_HIST];                       // w[i]: phase of lag i of the coming step (w[0] unused)
    double V[PER];
    int n = g.n_first;
    const int last = g.n_first + g.k - 1;
#pragma unroll
    for (int p = 0; p < PER; ++p) {
        u[p] = st[mode[p]];
#pragma unroll
        for (int j = 1; j <= MAX_HIST; ++j) {
            // (Vu)^ of step n - j, and the phase of its lag; lags before the start are not used
            const bool have = j <= g.order - 1 && n - j >= 0;
            r[p][j - 1] = have ? ring[(size_t)((n - j) % RS) * N + mode[p]] : make_double2(0.0, 0.0);
            w[p][j - 1] = have && j >= 2 ? factor(main_iv(n - j + 1), 0, mode[p]) : make_int4(0, 0, 0, 0);
        }
    }
    const double hmu0 = a.h * a.mu[0];
#pragma unroll 1
    for (; n <= last; ++n) {
        if (n <= g.S) {
            // start-up: L trapezoid chains of 1, 2, 4, .. sub-steps, Richardson combination
            double2 acc[PER];
#pragma unroll
            for (int p = 0; p < PER; ++p) acc[p] = make_double2(0.0, 0.0);
#pragma unroll 1
            for (int c = 0; c < g.L; ++c) {
                double2 x[PER], y[PER];
#pragma unroll
                for (int p = 0; p < PER; ++p) {
                    x[p] = u[p];
                    y[p] = r[p][0];
                }
                const double hc = 0.5 * (a.h / (double)(1 << c));
                const int len = 8 >> c;
#pragma unroll 1
                for (int i = 0; i < (1 << c); ++i) {
                    const int iv = (n - 1) * ((1 << g.L) - 1) + ((1 << c) - 1) + i;
                    potential(8 * (n - 1) + (i + 1) * len, V);
#pragma unroll
                    for (int p = 0; p < PER; ++p) {
                        double2 one[MAX_HIST];
#pragma unroll
                        for (int j = 0; j < MAX_HIST; ++j) one[j] = j == 0 ? y[p] : make_double2(0.0, 0.0);
                        const int4 w0 = factor(iv, c, mode[p]);
                        W[p] = fx_horner(x[p], one, 1, g.half_w, a.h_w, a.h_e - c, [&](int) { return w0; });
                    }
                    core<N>(W, V, hc, y, A, B, Q, tw);
#pragma unroll
                    for (int p = 0; p < PER; ++p) x[p] = update64(W[p], y[p], hc);
                }
#pragma unroll
                for (int p = 0; p < PER; ++p)
                    acc[p] = make_double2(fma(g.rich[c], x[p].x, acc[p].x), fma(g.rich[c], x[p].y, acc[p].y));
            }
#pragma unroll
            for (int p = 0; p < PER; ++p) u[p] = acc[p];
            potential(8 * n, V);
            core<N>(u, V, 0.0, R, A, B, Q, tw);
        } else {
            potential(8 * n, V);
#pragma unroll
            for (int p = 0; p < PER; ++p) {
                w[p][0] = factor(main_iv(n), 0, mode[p]);
                W[p] = fx_horner(u[p], r[p], g.order - 1, a.mu_w, a.h_w, a.h_e, [&](int i) { return w[p][i]; });
            }
            core<N>(W, V, hmu0, R, A, B, Q, tw);
#pragma unroll
            for (int p = 0; p < PER; ++p) u[p] = update64(W[p], R[p], hmu0);
        }
#pragma unroll
        for (int p = 0; p < PER; ++p) {
            if (n <= g.S) w[p][0] = factor(main_iv(n), 0, mode[p]);
#pragma unroll
            for (int j = MAX_HIST - 1; j >= 1; --j) {
                r[p][j] = r[p][j - 1];
                w[p][j] = w[p][j - 1];
            }
            r[p][0] = R[p];
            if (own) ring[(size_t)(n % RS) * N + mode[p]] = R[p];
        }
    }
#pragma unroll
    for (int p = 0; p < PER; ++p)
        if (own) st[mode[p]] = u[p];
}

template <int N>
cudaError_t go(const KArgs& a, const Run1DArgs& g, cudaStream_t s) {
    static DeviceOnce once;
    const cudaError_t e = once([] {
        return cudaFuncSetAttribute(k_run1d64<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Run1D64<N>::smem);
    });
    if (e != cudaSuccess) return e;
    k_run1d64<N><<<a.B, Run1D64<N>::T, Run1D64<N>::smem, s>>>(a, g);
    return cudaGetLastError();
}

}  // namespace

bool run1d64_supported(int n) { return n >= 8 && n <= RUN1D64_MAX && (n & (n - 1)) == 0; }

cudaError_t launch_run1d64(const KArgs& a, const Run1DArgs& g, cudaStream_t s) {
    switch (a.n0) {
        case 8: return go<8>(a, g, s);
        case 16: return go<16>(a, g, s);
        case 32: return go<32>(a, g, s);
        case 64: return go<64>(a, g, s);
        case 128: return go<128>(a, g, s);
        case 256: return go<256>(a, g, s);
        case 512: return go<512>(a, g, s);
        case 1024: return go<1024>(a, g, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace tdse
