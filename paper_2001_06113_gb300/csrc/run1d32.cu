// Runs of 1D mixed-precision Adams steps (interaction picture) in one launch,
// one CTA per instance, n = 8..8192: the loop over the steps is in the kernel.
//
// The step is that of step1d.cuh, operation for operation (same bits), with the
// state in registers from step to step and the history in the ring slots (L2;
// each thread reads back its own modes, so the steps need no barrier between
// them).  Bound by the latency of those loads and by issue (339 instructions per
// point and step).  2048 instances of 512 points, per step: one launch each 29.9,
// here 21.0 us.
//
// The start-up (lab frame, double-float) likewise: one launch runs the L
// Richardson chains of a start-up step, chain c of an instance its 2^c
// trapezoid sub-steps in one CTA, instead of 15 step launches and 8 copies.
// 2048 x 512 points, 7 start-up steps: 4.0 -> 2.3 ms.
#include "device_once.h"
#include "step_common.cuh"
#include "step1d.cuh"

namespace tdse {
namespace {

#ifndef RUN_THREADS
#define RUN_THREADS 1024
#endif
constexpr int RUN1D32_MAX = 8192;

template <int N> struct Run1D32 {
    static constexpr int T = N == 8192 ? 1024 : threads_1d(N);   // 8 modes per thread
    using FI = Fft<float2, N, 1, 1, T, true>;
    using FW = Fft<float2, N, 1, 1, T, false>;
    static constexpr int PB = FI::PF, RB = FI::RF;
    static constexpr size_t smem = (size_t)fft_len<float2>(N) * sizeof(float2);
    // 1024 threads per SM (64 registers): 512 (128 registers, nothing spilled) 22.2,
    // 640 23.3, 768 23.7, 1024 21.0 us per step of 2048 x 512 points; with the
    // history in shared memory (6 CTAs per SM) 26.5
    static constexpr int MINB = RUN_THREADS / T < 1 ? 1 : (RUN_THREADS / T > 32 ? 32 : RUN_THREADS / T);
    static constexpr int MINB_START = 512 / T < 1 ? 1 : (512 / T > 16 ? 16 : 512 / T);   // 128 registers
};
template <int T> struct GroupOf {
    using type = CtaSync;
};
template <> struct GroupOf<32> {
    using type = WarpSync;
};

template <int N>
__global__ void __launch_bounds__(Run1D32<N>::T, Run1D32<N>::MINB) k_run1d32(const __grid_constant__ KArgs a,
                                                                            const __grid_constant__ Run1DArgs g,
                                                                            const float* __restrict__ wtab) {
    using G = Run1D32<N>;
    using FI = typename G::FI;
    using FW = typename G::FW;
    constexpr int PB = G::PB, RB = G::RB, T = G::T;
    static_assert(FI::RL == FW::RF && FI::PL == FW::PF && FW::RL == RB && FW::PL == PB, "a thread keeps its modes");
    static_assert(PB * RB <= 8, "the state fits the registers");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* buf = reinterpret_cast<float2*>(smem_raw);
    __shared__ float4 wsm[2][CL_TAB / 4];
    const typename GroupOf<T>::type sync{};
    const int b = blockIdx.x, tid = threadIdx.x;
    float4* st = reinterpret_cast<float4*>(a.uhat) + (size_t)b * N;
    float2* ring = reinterpret_cast<float2*>(a.ring) + (size_t)b * a.ring_slots * N;
    const int RS = a.ring_slots, nhist = g.order - 1;
    const float2 *tw = a.tw32_0, *twl = a.tw32lo_0;
    const float scale = 1.0f / (float)N, hmu0 = (float)(a.h * a.mu[0]);
    const double* tfac = a.tfac + (size_t)b * a.ntf;
    const float2* V0f = a.V0f + (size_t)b * a.vstride;
    auto own = [&](int p, int r, int& k) {      // mode k of (p, r); false where this thread has none
        int j, line;
        const bool ok = FI::item(p, FI::NBF, j, line, tid);
        k = j + r * FI::NBF;
        return ok;
    };
    float4 v[PB][RB];
#pragma unroll
    for (int p = 0; p < PB; ++p)
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            int k;
            if (!own(p, r, k)) continue;
            v[p][r] = st[k];
        }
    const int last = g.n_first + g.k - 1;
    for (int i = tid; i < CL_TAB / 4; i += T) wsm[g.n_first & 1][i] = reinterpret_cast<const float4*>(wtab)[(size_t)g.n_first * (CL_TAB / 4) + i];
    sync();
#pragma unroll 1
    for (int n = g.n_first; n <= last; ++n) {
        const float* w = reinterpret_cast<const float*>(wsm[n & 1]);
        float2 E[PB][RB], in[PB][RB], mid[FI::PL][FI::RL];
        {
            float2 S[PB][RB];
#pragma unroll
            for (int p = 0; p < PB; ++p)
#pragma unroll
                for (int r = 0; r < RB; ++r) S[p][r] = make_float2(0.f, 0.f);
            int slot = (n - nhist) % RS;
#pragma unroll 1
            for (int j = nhist; j >= 1; --j) {
                const float4 c = make_float4(w[6 + 4 * (j - 1)], w[7 + 4 * (j - 1)], w[8 + 4 * (j - 1)], w[9 + 4 * (j - 1)]);
#pragma unroll
                for (int p = 0; p < PB; ++p)
#pragma unroll
                    for (int r = 0; r < RB; ++r) {
                        int k;
                        if (own(p, r, k)) S[p][r] = ip_add_lag(c, ring[(size_t)slot * N + k], S[p][r]);
                    }
                slot = slot + 1 == RS ? 0 : slot + 1;
            }
#pragma unroll
            for (int p = 0; p < PB; ++p)
#pragma unroll
                for (int r = 0; r < RB; ++r) {
                    int k;
                    if (!own(p, r, k)) continue;
                    v[p][r] = ff_minus_i_times(v[p][r], a.h_hi, a.h_lo, S[p][r]);
                    E[p][r] = e_1d(a, b, n, k);
                    in[p][r] = cmul(E[p][r], make_float2(v[p][r].x, v[p][r].y));
                }
        }
        FI::run(in, mid, buf, tw, twl, tid, sync);
        if constexpr (FI::NPASS == 1) sync();
        // The next step's weights: past the transform's barriers every thread has
        // left the step before, the last to read their buffer.  The forward
        // transform's barriers publish them (n = 8 has none: one of its own).
        if (n < last)
            for (int i = tid; i < CL_TAB / 4; i += T)
                wsm[(n + 1) & 1][i] = __ldg(reinterpret_cast<const float4*>(wtab) + (size_t)(n + 1) * (CL_TAB / 4) + i);
        if constexpr (FW::NPASS == 1) sync();
        const double vfac = tfac[8 * (size_t)n];
        const float fh = (float)vfac, fl = (float)(vfac - (double)fh);
        const float2* V = V0f + (g.vtable ? (size_t)(8 * g.S_eff + (n - g.S_eff)) * N : 0);
#pragma unroll
        for (int p = 0; p < FI::PL; ++p) {
            int j, line;
            if (FI::item(p, FI::NBL, j, line, tid)) {
#pragma unroll
                for (int r = 0; r < FI::RL; ++r) {
                    const float2 v2 = V[j + r * FI::NBL];
                    const float vh = fh * v2.x;
                    const float vl = fmaf(fh, v2.x, -vh) + fmaf(fh, v2.y, fl * v2.x);
                    mid[p][r] = implicit_solve_times_V(mid[p][r], vh, vl, hmu0);
                }
            }
        }
        FW::run(mid, in, buf, tw, twl, tid, sync);
        const float2 z = make_float2(w[0], w[1]);
        const float4 d = make_float4(w[2], w[3], w[4], w[5]);
        const int out = n % RS;
#pragma unroll
        for (int p = 0; p < PB; ++p)
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                int k;
                if (!own(p, r, k)) continue;
                const float2 rv = cmul(z, cmul(conjf2(E[p][r]), cscale(in[p][r], scale)));
                ring[(size_t)out * N + k] = rv;
                v[p][r] = ip_update(d, v[p][r], rv);
            }
    }
#pragma unroll
    for (int p = 0; p < PB; ++p)
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            int k;
            if (!own(p, r, k)) continue;
            st[k] = v[p][r];
        }
}

template <int N>
__global__ void __launch_bounds__(Run1D32<N>::T, Run1D32<N>::MINB_START) k_start1d32(const __grid_constant__ KArgs a,
                                                                              const __grid_constant__ Start1DArgs g) {
    using G = Run1D32<N>;
    using FI = typename G::FI;
    using FW = typename G::FW;
    constexpr int PB = G::PB, RB = G::RB, T = G::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* buf = reinterpret_cast<float2*>(smem_raw);
    const typename GroupOf<T>::type sync{};
    const int b = blockIdx.x, c = g.L - 1 - blockIdx.y, tid = threadIdx.x;       // the longest chain first
    const float4* st = reinterpret_cast<const float4*>(a.uhat) + (size_t)b * N;
    const float2* r0 = reinterpret_cast<const float2*>(a.ring) + ((size_t)b * a.ring_slots + g.slot) * N;
    float4* dst = g.chains + ((size_t)c * a.B + b) * N;
    const float2 *tw = a.tw32_0, *twl = a.tw32lo_0;
    const float scale = 1.0f / (float)N, hmu0 = (float)g.hmu0[c];
    const double* tfac = a.tfac + (size_t)b * a.ntf;
    const float2* V0f = a.V0f + (size_t)b * a.vstride;
    const float4* adv = a.advff + (size_t)b * a.n_int * (size_t)(a.nh + a.nl);
    auto own = [&](int p, int r, int& k) {
        int j, line;
        const bool ok = FI::item(p, FI::NBF, j, line, tid);
        k = j + r * FI::NBF;
        return ok;
    };
    float4 v[PB][RB];
    float2 rv[PB][RB];
#pragma unroll
    for (int p = 0; p < PB; ++p)
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            int k;
            if (!own(p, r, k)) continue;
            v[p][r] = st[k];
            rv[p][r] = r0[k];
        }
    KArgs w{};                                   // the sub-step's weights, for the shared update
    w.hmu0_hi = g.hmu0_hi[c];
    w.hmu0_lo = g.hmu0_lo[c];
#pragma unroll 1
    for (int i = 0; i < (1 << c); ++i) {
        const float4* q = adv + (size_t)(g.interval0 + (1 << c) - 1 + i) * (size_t)(a.nh + a.nl);
        const int tf = g.tf0 + (i + 1) * (8 >> c);
        float2 in[PB][RB], mid[FI::PL][FI::RL];
#pragma unroll
        for (int p = 0; p < PB; ++p)
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                int k;
                if (!own(p, r, k)) continue;
                // the sum of one lag, weight 1/2 (its low part is zero), as history_sum_f32
                const float2 S = make_float2(fmaf(0.5f, rv[p][r].x, 0.f), fmaf(0.5f, rv[p][r].y, 0.f));
                const float4 X = ff_minus_i_times(v[p][r], g.h_hi[c], g.h_lo[c], S);
                const float4 kin = __ldg(&a.kinff[(size_t)c * N + k]);
                const float4 ph = ffc_mul(kin, ffc_mul(__ldg(&q[k >> a.lb]), __ldg(&q[a.nh + (k & (a.nl - 1))])));
                v[p][r] = ffc_mul(ph, X);
                in[p][r] = st_to_c<float2>(v[p][r]);
            }
        FI::run(in, mid, buf, tw, twl, tid, sync);
        const double vfac = tfac[tf];
        const float fh = (float)vfac, fl = (float)(vfac - (double)fh);
        const float2* V = V0f + (g.vtable ? (size_t)tf * N : 0);
#pragma unroll
        for (int p = 0; p < FI::PL; ++p) {
            int j, line;
            if (FI::item(p, FI::NBL, j, line, tid)) {
#pragma unroll
                for (int r = 0; r < FI::RL; ++r) {
                    const float2 v2 = V[j + r * FI::NBL];
                    const float vh = fh * v2.x;
                    const float vl = fmaf(fh, v2.x, -vh) + fmaf(fh, v2.y, fl * v2.x);
                    mid[p][r] = implicit_solve_times_V(mid[p][r], vh, vl, hmu0);
                }
            }
        }
        FW::run(mid, in, buf, tw, twl, tid, sync);
#pragma unroll
        for (int p = 0; p < PB; ++p)
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                int k;
                if (!own(p, r, k)) continue;
                rv[p][r] = cscale(in[p][r], scale);
                v[p][r] = update_ff(w, v[p][r], rv[p][r]);
            }
    }
#pragma unroll
    for (int p = 0; p < PB; ++p)
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            int k;
            if (own(p, r, k)) dst[k] = v[p][r];
        }
}

template <int N>
cudaError_t prepare() {
    static DeviceOnce once;
    auto attributes = [](auto kernel) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Run1D32<N>::smem);
        return e != cudaSuccess ? e : cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                                           cudaSharedmemCarveoutMaxShared);
    };
    return once([&] {
        const cudaError_t e = attributes(k_run1d32<N>);
        return e != cudaSuccess ? e : attributes(k_start1d32<N>);
    });
}
template <int N>
cudaError_t start(const KArgs& a, const Start1DArgs& g, cudaStream_t s) {
    const cudaError_t e = prepare<N>();
    if (e != cudaSuccess) return e;
    k_start1d32<N><<<dim3(a.B, g.L), Run1D32<N>::T, Run1D32<N>::smem, s>>>(a, g);
    return cudaGetLastError();
}
template <int N>
cudaError_t go(const KArgs& a, const Run1DArgs& g, const float* wtab, cudaStream_t s) {
    const cudaError_t e = prepare<N>();
    if (e != cudaSuccess) return e;
    k_run1d32<N><<<a.B, Run1D32<N>::T, Run1D32<N>::smem, s>>>(a, g, wtab);
    return cudaGetLastError();
}

}  // namespace

bool run1d32_supported(int n) { return n >= 8 && n <= RUN1D32_MAX && (n & (n - 1)) == 0; }

#define TDSE_RUN32(CALL)                  \
    switch (n) {                          \
        case 8: return CALL(8);           \
        case 16: return CALL(16);         \
        case 32: return CALL(32);         \
        case 64: return CALL(64);         \
        case 128: return CALL(128);       \
        case 256: return CALL(256);       \
        case 512: return CALL(512);       \
        case 1024: return CALL(1024);     \
        case 2048: return CALL(2048);     \
        case 4096: return CALL(4096);     \
        case 8192: return CALL(8192);     \
        default: return cudaErrorInvalidValue; \
    }
cudaError_t run1d32_prepare(int n) {
#define TDSE_P(N) prepare<N>()
    TDSE_RUN32(TDSE_P)
}
cudaError_t launch_start1d32(const KArgs& a, const Start1DArgs& g, cudaStream_t s) {
    const int n = a.n0;
#define TDSE_S(N) start<N>(a, g, s)
    TDSE_RUN32(TDSE_S)
}
cudaError_t launch_run1d32(const KArgs& a, const Run1DArgs& g, const float* wtab, cudaStream_t s) {
    const int n = a.n0;
#define TDSE_G(N) go<N>(a, g, wtab, s)
    TDSE_RUN32(TDSE_G)
}

}  // namespace tdse
