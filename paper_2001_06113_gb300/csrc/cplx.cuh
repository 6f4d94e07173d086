// Complex arithmetic on double2/float2 and a shared-memory Stockham FFT (FP32
// values as written below; FP64 values through the same passes in 64-bit fixed
// point, fx.cuh).
//
// The FFT computes, for each of L interleaved sequences of length N,
//     forward:  X_k = sum_j x_j e^{-2 pi i j k / N}
//     inverse:  x_j = sum_k X_k e^{+2 pi i j k / N}     (no 1/N)
// as a Stockham auto-sort sequence of passes.  In pass s with Ns = product of
// the earlier radices, butterfly j (0 <= j < N/R) reads x[j + r N/R], twiddles
// by e^{-+2 pi i (j mod Ns) r / (Ns R)}, takes an R-point DFT in registers and
// writes positions (j - j mod Ns) R + j mod Ns + r Ns.  The passes are radix 8
// plus one radix-2 or radix-4 pass when log2 N is not a multiple of 3 (second
// of three or more passes; with two passes first for forward transforms, last
// for inverse ones).  Then the last pass of a
// transform writes exactly the positions j + r N/R that the first pass of the
// next transform reads, so a transform's inputs and outputs stay in the
// registers of the thread that owns them: the first pass starts from
// registers, the last pass ends in registers, and the epilogue/prologue work of
// the step (history sum, implicit solve, mode update) runs there.  Shared
// memory holds element (pos, line) at buf[pos * PS + line], consecutive threads
// taking consecutive lines (interleaved columns).  Twiddles come from a global table
// tw[m] = e^{-2 pi i m / N} (read through the read-only cache); in FP32 a
// second table twlo = e^{-2 pi i m/N} - tw holds the rounding residual, used
// (v tw + v twlo) when TDSE_TWIDDLE_LO is set.
#pragma once
#include <cuda_runtime.h>

#include "fx.cuh"

namespace tdse {

// Real type, and the type of a twiddle table's entries: FP64 transforms run
// in 64-bit fixed point (fx.cuh).
template <class C> struct cx_traits;
template <> struct cx_traits<double2> { using real = double; using tw = int4; };
template <> struct cx_traits<float2> { using real = float; using tw = float2; };
template <class C> using tw_t = typename cx_traits<C>::tw;

__device__ __forceinline__ double2 operator+(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 operator-(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 operator+(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 operator-(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cscale(double2 a, double s) { return make_double2(a.x * s, a.y * s); }
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }

template <class D> __device__ __forceinline__ D cvt(double2 a);
template <> __device__ __forceinline__ double2 cvt<double2>(double2 a) { return a; }
template <> __device__ __forceinline__ float2 cvt<float2>(double2 a) { return make_float2((float)a.x, (float)a.y); }
template <class D> __device__ __forceinline__ D cvt(float2 a);
template <> __device__ __forceinline__ double2 cvt<double2>(float2 a) { return make_double2(a.x, a.y); }
template <> __device__ __forceinline__ float2 cvt<float2>(float2 a) { return a; }

template <class C> __device__ __forceinline__ C czero();
template <> __device__ __forceinline__ double2 czero<double2>() { return make_double2(0.0, 0.0); }
template <> __device__ __forceinline__ float2 czero<float2>() { return make_float2(0.f, 0.f); }

// multiply by -i (forward) or +i (inverse)
template <bool INV, class C> FX_HD C rot90(C a) {
    C r;
    if (INV) { r.x = -a.y; r.y = a.x; } else { r.x = a.y; r.y = -a.x; }
    return r;
}

// multiply by e^{-+ i pi/4} = (1 -+ i)/sqrt(2).  In FP32 the constant is
// applied as hi + lo so that the butterfly has no fixed rounding of 1/sqrt(2)
// (a rounding repeated identically at every step would bias the transform).
template <bool INV> FX_HD longlong2 rot45(longlong2 a) {
    const long long u = INV ? a.x - a.y : a.x + a.y, v = INV ? a.x + a.y : a.y - a.x;
    return make_longlong2(fx_times_rsqrt2(u), fx_times_rsqrt2(v));
}
template <bool INV> __device__ __forceinline__ float2 rot45(float2 a) {
    const float sh = 0.707106769084930419921875f;          // float(1/sqrt 2)
    const float sl = 1.2101617485882343317e-08f;           // 1/sqrt 2 - sh
    const float u = INV ? a.x - a.y : a.x + a.y;
    const float v = INV ? a.x + a.y : a.y - a.x;
    return make_float2(fmaf(u, sh, u * sl), fmaf(v, sh, v * sl));
}

template <bool INV, class C> FX_HD void dft2(C* v) {
    C t = v[0] - v[1]; v[0] = v[0] + v[1]; v[1] = t;
}

template <bool INV, class C> FX_HD void dft4(C& a0, C& a1, C& a2, C& a3) {
    C t0 = a0 + a2, t1 = a0 - a2, t2 = a1 + a3, t3 = rot90<INV>(a1 - a3);
    a0 = t0 + t2; a2 = t0 - t2; a1 = t1 + t3; a3 = t1 - t3;
}

template <bool INV, class C> FX_HD void dft8(C* v) {
    C e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    C o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4<INV>(e0, e1, e2, e3);
    dft4<INV>(o0, o1, o2, o3);
    o1 = rot45<INV>(o1);
    o2 = rot90<INV>(o2);
    o3 = rot90<INV>(rot45<INV>(o3));
    v[0] = e0 + o0; v[4] = e0 - o0;
    v[1] = e1 + o1; v[5] = e1 - o1;
    v[2] = e2 + o2; v[6] = e2 - o2;
    v[3] = e3 + o3; v[7] = e3 - o3;
}

template <int R, bool INV, class C> FX_HD void dft_r(C* v) {
    if constexpr (R == 2) dft2<INV>(v);
    else if constexpr (R == 4) dft4<INV>(v[0], v[1], v[2], v[3]);
    else dft8<INV>(v);
}

constexpr int ilog2(int n) { return n <= 1 ? 0 : 1 + ilog2(n / 2); }


template <int N, bool INV> struct FftPlan {
    static constexpr int P = ilog2(N);
    static constexpr int RS = (P % 3 == 0) ? 8 : (1 << (P % 3));
    static constexpr int NPASS = (P % 3 == 0) ? P / 3 : P / 3 + 1;
    // Boundary passes are radix 8 whenever possible (small radix in the second
    // pass), so that a thread owns 8 values per item at both ends; with only two
    // passes the small radix goes first (forward) / last (inverse).
    static constexpr int radix(int s) {
        return RS == 8 ? 8 : (NPASS >= 3 ? (s == 1 ? RS : 8) : ((INV ? (s == NPASS - 1) : (s == 0)) ? RS : 8));
    }
    static constexpr int ns(int s) { return s == 0 ? 1 : ns(s - 1) * radix(s - 1); }
};

// Radix-4 passes (and one radix-2 pass, placed as above) for transforms whose
// latency counts: half the work and registers per thread of a radix-8 pass.
template <int N, bool INV> struct FftPlan4 {
    static constexpr int P = ilog2(N);
    static constexpr int NPASS = (P + 1) / 2;
    static constexpr int radix(int s) {
        return P % 2 == 0 ? 4 : (NPASS >= 3 ? (s == 1 ? 2 : 4) : ((INV ? (s == NPASS - 1) : (s == 0)) ? 2 : 4));
    }
    static constexpr int ns(int s) { return s == 0 ? 1 : ns(s - 1) * radix(s - 1); }
};

// v * w (w from tw, conjugated for the inverse).
// TDSE_TWIDDLE_LO = 1 applies the FP32 twiddle as hi + lo.  Off by default:
// on the 512^2 mixed workload it lowers the 2000-step error from 5.1e-7 to
// 4.4e-7 at a 7% cost in step time.
#ifndef TDSE_TWIDDLE_LO
#define TDSE_TWIDDLE_LO 0
#endif
template <bool INV> __device__ __forceinline__ float2 twiddle(float2 v, const float2* __restrict__ tw,
                                                              const float2* __restrict__ twl, int idx) {
    float2 w = __ldg(&tw[idx]);
    if (!TDSE_TWIDDLE_LO) {
        if (INV) w.y = -w.y;
        return cmul(v, w);
    }
    float2 wl = __ldg(&twl[idx]);
    if (INV) { w.y = -w.y; wl.y = -wl.y; }
    float2 t = cmul(v, w);
    t.x = fmaf(v.x, wl.x, fmaf(-v.y, wl.y, t.x));
    t.y = fmaf(v.x, wl.y, fmaf(v.y, wl.x, t.y));
    return t;
}

// Barrier policies for a group of threads that runs one transform: the whole
// CTA, one warp, or a named barrier over n threads (a multiple of 32) when
// several groups share a CTA.
struct CtaSync {
    __device__ __forceinline__ void operator()() const { __syncthreads(); }
};
struct WarpSync {
    __device__ __forceinline__ void operator()() const { __syncwarp(); }
};
struct GroupSync {
    unsigned id, n;
    __device__ __forceinline__ void operator()() const { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
};

// L interleaved length-N transforms by T threads (thread index tid in 0..T-1
// of the group, barrier `sync`); element (pos, line) at buf[pos * PS + line].
// Item it of a pass with NB butterflies is butterfly j = it / L of line it % L.
template <int N, int L, int T, bool INV>
struct FftShape {
    using Plan = FftPlan<N, INV>;
    static constexpr int NPASS = Plan::NPASS;
    static constexpr int RF = Plan::radix(0);
    static constexpr int RL = Plan::radix(NPASS - 1);
    static constexpr int NBF = N / RF;           // first pass: item (j, line) owns positions j + r NBF
    static constexpr int NBL = N / RL;           // last pass:  item (j, line) owns positions j + r NBL
    static constexpr int PF = (NBF * L + T - 1) / T;
    static constexpr int PL = (NBL * L + T - 1) / T;

    __device__ static __forceinline__ bool item(int p, int NB, int& j, int& line, int tid) {
        const int it = tid + p * T;
        line = it % L;
        j = it / L;
        return ((NB * L) % T == 0) || it < NB * L;
    }
};

// Buffer elements of a single padded line of N points (FP64: not padded).
template <class C> constexpr int fft_len(int n) { return sizeof(C) == 8 ? n + n / 16 : n; }

template <class C, int N, int L, int PS, int T, bool INV>
struct Fft : FftShape<N, L, T, INV> {
    using Shape = FftShape<N, L, T, INV>;
    using Plan = FftPlan<N, INV>;
    using Shape::item;
    using Shape::NBF;
    using Shape::NBL;
    using Shape::NPASS;
    using Shape::PF;
    using Shape::PL;
    using Shape::RF;
    using Shape::RL;

    // Element (pos, line) of the buffer.  A single line is padded by one element
    // in 16: without it the stride-8 stores of the first pass meet in two of
    // 16 banks (192 -> 72 shared-memory cycles per butterfly of a 512-point
    // line); fft_len(N) elements in all.
    __device__ static __forceinline__ int at(int pos, int line) {
        return L == 1 && PS == 1 ? pos + (pos >> 4) : pos * PS + line;
    }

    template <int S, class Sync>
    __device__ static __forceinline__ void mid_pass(C* buf, const C* __restrict__ tw, const C* __restrict__ twl,
                                                    int tid, const Sync& sync) {
        constexpr int R = Plan::radix(S);
        constexpr int Ns = Plan::ns(S);
        constexpr int NB = N / R;
        constexpr int PER = (NB * L + T - 1) / T;
        C v[PER][R];
#pragma unroll
        for (int p = 0; p < PER; ++p) {
            int j, line;
            if (item(p, NB, j, line, tid)) {
#pragma unroll
                for (int r = 0; r < R; ++r) v[p][r] = buf[at(j + r * NB, line)];
            }
        }
        sync();
#pragma unroll
        for (int p = 0; p < PER; ++p) {
            int j, line;
            if (item(p, NB, j, line, tid)) {
                const int k = j & (Ns - 1);
                constexpr int stride = N / (Ns * R);
#pragma unroll
                for (int r = 1; r < R; ++r) v[p][r] = twiddle<INV>(v[p][r], tw, twl, k * r * stride);
                dft_r<R, INV>(v[p]);
                const int base = (j - k) * R + k;
#pragma unroll
                for (int r = 0; r < R; ++r) buf[at(base + r * Ns, line)] = v[p][r];
            }
        }
        sync();
    }

    template <int S, class Sync>
    __device__ static __forceinline__ void mids(C* buf, const C* __restrict__ tw, const C* __restrict__ twl, int tid,
                                                const Sync& sync) {
        if constexpr (S <= NPASS - 2) {
            mid_pass<S>(buf, tw, twl, tid, sync);
            mids<S + 1>(buf, tw, twl, tid, sync);
        }
    }

    // in[p][r]: value at position j + r NBF of the item (p); out[p][r]: result at
    // position j + r NBL.  buf must not be in use by any thread of the group on
    // entry; the call ends with a barrier (buf free again).
    template <class Sync>
    __device__ static __forceinline__ void run(C (&in)[PF][RF], C (&out)[PL][RL], C* buf,
                                               const C* __restrict__ tw, const C* __restrict__ twl, int tid,
                                               const Sync& sync) {
        if constexpr (NPASS == 1) {
#pragma unroll
            for (int p = 0; p < PF; ++p) {
                dft_r<RF, INV>(in[p]);
#pragma unroll
                for (int r = 0; r < RF; ++r) out[p][r] = in[p][r];
            }
        } else {
#pragma unroll
            for (int p = 0; p < PF; ++p) {
                int j, line;
                if (item(p, NBF, j, line, tid)) {
                    dft_r<RF, INV>(in[p]);
#pragma unroll
                    for (int r = 0; r < RF; ++r) buf[at(j * RF + r, line)] = in[p][r];
                }
            }
            sync();
            mids<1>(buf, tw, twl, tid, sync);
#pragma unroll
            for (int p = 0; p < PL; ++p) {
                int j, line;
                if (item(p, NBL, j, line, tid)) {
#pragma unroll
                    for (int r = 0; r < RL; ++r) out[p][r] = buf[at(j + r * NBL, line)];
#pragma unroll
                    for (int r = 1; r < RL; ++r) out[p][r] = twiddle<INV>(out[p][r], tw, twl, j * r);
                    dft_r<RL, INV>(out[p]);
                }
            }
            sync();
        }
    }

    // The same transform split for callers that produce the inputs / consume
    // the outputs one item at a time in a non-unrolled loop (NPASS > 1):
    //   first_item(p, v)  for every p, then  middle(...),  then either
    //   last_item(p, v)   for every p followed by  finish(sync)   (buf free again).
    __device__ static __forceinline__ void first_item(int p, C (&v)[RF], C* buf, int tid) {
        int j, line;
        if (item(p, NBF, j, line, tid)) {
            dft_r<RF, INV>(v);
#pragma unroll
            for (int r = 0; r < RF; ++r) buf[at(j * RF + r, line)] = v[r];
        }
    }
    template <class Sync>
    __device__ static __forceinline__ void middle(C* buf, const C* __restrict__ tw, const C* __restrict__ twl,
                                                  int tid, const Sync& sync) {
        sync();
        mids<1>(buf, tw, twl, tid, sync);
    }
    __device__ static __forceinline__ bool last_item(int p, C (&v)[RL], const C* buf, const C* __restrict__ tw,
                                                     const C* __restrict__ twl, int tid, int& j) {
        int line;
        if (!item(p, NBL, j, line, tid)) return false;
#pragma unroll
        for (int r = 0; r < RL; ++r) v[r] = buf[at(j + r * NBL, line)];
#pragma unroll
        for (int r = 1; r < RL; ++r) v[r] = twiddle<INV>(v[r], tw, twl, j * r);
        dft_r<RL, INV>(v);
        return true;
    }
    template <class Sync>
    __device__ static __forceinline__ void finish(const Sync& sync) { sync(); }
};

// ---------------------------------------------------------------------------
// L interleaved length-N transforms done in place by a whole CTA of T threads:
// element (pos, line) at buf[pos * LS + line], consecutive threads taking
// consecutive lines.  Each pass loads all butterflies of the thread into
// registers, synchronises, then writes (in place).  The caller must have
// synchronised after filling buf; the call ends with a barrier.
template <class C, int N, int L, int LS, int T, bool INV>
struct CtaFft {
    using Plan = FftPlan<N, INV>;
    template <int S>
    __device__ static __forceinline__ void pass(C* buf, const C* __restrict__ tw, const C* __restrict__ twl) {
        if constexpr (S < Plan::NPASS) {
            constexpr int R = Plan::radix(S);
            constexpr int Ns = Plan::ns(S);
            constexpr int NB = N / R;
            constexpr int ITEMS = NB * L;
            constexpr int PER = (ITEMS + T - 1) / T;
            C v[PER][R];
#pragma unroll
            for (int p = 0; p < PER; ++p) {
                const int it = threadIdx.x + p * T;
                if (ITEMS % T == 0 || it < ITEMS) {
                    const int line = it % L, j = it / L;
#pragma unroll
                    for (int r = 0; r < R; ++r) v[p][r] = buf[(j + r * NB) * LS + line];
                }
            }
            __syncthreads();
#pragma unroll
            for (int p = 0; p < PER; ++p) {
                const int it = threadIdx.x + p * T;
                if (ITEMS % T == 0 || it < ITEMS) {
                    const int line = it % L, j = it / L;
                    const int k = j & (Ns - 1);
                    constexpr int stride = N / (Ns * R);
                    if (Ns > 1) {
#pragma unroll
                        for (int r = 1; r < R; ++r) v[p][r] = twiddle<INV>(v[p][r], tw, twl, k * r * stride);
                    }
                    dft_r<R, INV>(v[p]);
                    const int base = (j - k) * R + k;
#pragma unroll
                    for (int r = 0; r < R; ++r) buf[(base + r * Ns) * LS + line] = v[p][r];
                }
            }
            __syncthreads();
            pass<S + 1>(buf, tw, twl);
        }
    }
    __device__ static __forceinline__ void run(C* buf, const C* __restrict__ tw, const C* __restrict__ twl) {
        pass<0>(buf, tw, twl);
    }
};

// ---------------------------------------------------------------------------
// The same two transforms for FP64 values, in 64-bit fixed point (fx.cuh): tw
// holds int4 table factors, buf holds FP64 values outside a transform and
// integers inside.  The results are multiplied by 2^lg on the way out (exact).
//
// Pass S of radix R with its butterflies' values in v: twiddle and 1/R for
// S > 0, then the R-point DFT.
template <int N, bool INV, class PlanT = FftPlan<N, INV>>
struct FxPass {
    using Plan = PlanT;
    static constexpr int S0 = 62 - ilog2(Plan::radix(0));       // input scale
    static constexpr int GAIN = ilog2(N / Plan::radix(0));      // the passes' 1/R
    template <int S>
    FX_HD static void butterfly(longlong2* v, int j, const int4* __restrict__ tw) {
        constexpr int R = Plan::radix(S);
        if constexpr (S > 0) {
            constexpr int Ns = Plan::ns(S), LR = ilog2(R), stride = N / (Ns * R);
            const int k = j & (Ns - 1);
            v[0].x = (v[0].x + (1ll << (LR - 1))) >> LR;
            v[0].y = (v[0].y + (1ll << (LR - 1))) >> LR;
#pragma unroll
            for (int r = 1; r < R; ++r) v[r] = fx_mul<INV, 3 - LR>(v[r], fx_ldg(&tw[k * r * stride]));
        }
        dft_r<R, INV>(v);
    }
    // A pass divides by its radix whether or not its sums grew: an input in few
    // places (a smooth state's modes on a fine grid, a narrow state) would lose
    // log2(N / radix(0)) of its 59 bits.  Up to N = 1024 what is left is no less than
    // FP64 gives; longer lines are scaled up before each middle pass by what their
    // largest component leaves free (2^s, taken off the results' exponent).
    static constexpr bool rescales(int S) { return N >= 2048 && S > 0 && S < Plan::NPASS - 1; }
    FX_HD static unsigned magnitude(longlong2 v) {
        const int x = (int)(v.x >> 32), y = (int)(v.y >> 32);
        const unsigned a = (unsigned)(x ^ (x >> 31)), b = (unsigned)(y ^ (y >> 31));
        return a > b ? a : b;
    }
    FX_HD static int headroom(unsigned mag) {       // components below 2^62 after v 2^s
#ifdef __CUDA_ARCH__
        const int z = __clz((int)mag);
#else
        const int z = mag ? __builtin_clz(mag) : 32;
#endif
        return z > 2 ? z - 2 : 0;
    }
    FX_HD static longlong2 up(longlong2 v, int s) {
        return make_longlong2((long long)((unsigned long long)v.x << s), (long long)((unsigned long long)v.y << s));
    }
    // exponent of the results for block exponent E (of the largest high word mx)
    FX_HD static int out_exp(unsigned mx, int E, int lg) {
        return mx >= 0x7ff00000u ? FX_NAN : E - 1022 - S0 + GAIN + lg;
    }
};

// v 2^s for the block's common headroom s, which is returned; with the barrier that a
// pass needs between its loads and its stores.
template <class Fx, int T, int PER, int R, class Sync>
__device__ __forceinline__ int fx_rescale(longlong2 (&v)[PER][R], const Sync& sync) {
    __shared__ unsigned mx[T / 32];
    unsigned m = 0;
#pragma unroll
    for (int p = 0; p < PER; ++p)
#pragma unroll
        for (int r = 0; r < R; ++r) m = max(m, Fx::magnitude(v[p][r]));
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) mx[threadIdx.x >> 5] = m;
    sync();
    const int s = Fx::headroom(__reduce_max_sync(0xffffffffu, mx[(threadIdx.x & 31) % (T / 32)]));
#pragma unroll
    for (int p = 0; p < PER; ++p)
#pragma unroll
        for (int r = 0; r < R; ++r) v[p][r] = Fx::up(v[p][r], s);
    return s;
}

template <int N, int L, int LS, int T, bool INV>
struct CtaFft<double2, N, L, LS, T, INV> {
    using Fx = FxPass<N, INV>;
    using Plan = FftPlan<N, INV>;
    template <int S>
    __device__ static __forceinline__ void pass(longlong2* buf, const int4* __restrict__ tw, int X) {
        if constexpr (S < Plan::NPASS) {
            constexpr int R = Plan::radix(S), Ns = Plan::ns(S), NB = N / R, ITEMS = NB * L, PER = (ITEMS + T - 1) / T;
            longlong2 v[PER][R];
#pragma unroll
            for (int p = 0; p < PER; ++p) {
                const int it = threadIdx.x + p * T;
                if (ITEMS % T == 0 || it < ITEMS) {
#pragma unroll
                    for (int r = 0; r < R; ++r) v[p][r] = buf[(it / L + r * NB) * LS + it % L];
                }
            }
            if constexpr (Fx::rescales(S)) {
                static_assert(ITEMS % T == 0 && L == 1, "every value is set, one line");
                X -= fx_rescale<Fx, T>(v, CtaSync{});
            } else {
                __syncthreads();
            }
            store<S, PER, R, Ns>(buf, tw, v, X);
            __syncthreads();
            pass<S + 1>(buf, tw, X);
        }
    }
    template <int S, int PER, int R, int Ns>
    __device__ static __forceinline__ void store(longlong2* buf, const int4* __restrict__ tw, longlong2 (&v)[PER][R],
                                                 int X) {
        constexpr int ITEMS = N / R * L;
#pragma unroll
        for (int p = 0; p < PER; ++p) {
            const int it = threadIdx.x + p * T;
            if (ITEMS % T == 0 || it < ITEMS) {
                const int line = it % L, j = it / L, k = j & (Ns - 1);
                Fx::template butterfly<S>(v[p], j, tw);
                longlong2* out = buf + ((j - k) * R + k) * LS + line;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    if constexpr (S == Plan::NPASS - 1) reinterpret_cast<double2*>(out)[r * Ns * LS] = fx_to(v[p][r], X);
                    else out[r * Ns * LS] = v[p][r];
                }
            }
        }
    }
    __device__ static __forceinline__ void run(double2* dbuf, const int4* __restrict__ tw, const int4*, int lg = 0) {
        constexpr int R = Plan::radix(0), NB = N / R, ITEMS = NB * L, PER = (ITEMS + T - 1) / T;
        longlong2* buf = reinterpret_cast<longlong2*>(dbuf);
        double2 x[PER][R];
        unsigned mx = 0;
#pragma unroll
        for (int p = 0; p < PER; ++p) {
            const int it = threadIdx.x + p * T;
            if (ITEMS % T == 0 || it < ITEMS) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    x[p][r] = dbuf[(it / L + r * NB) * LS + it % L];
                    mx = max(mx, fx_hi(x[p][r]));
                }
            }
        }
        static_assert(T % L == 0, "a thread keeps its line");
        mx = fx_line_max<T, L>(mx);             // its barrier also orders the loads above before the stores below
        if constexpr (T <= 32) __syncwarp();
        const int E = fx_exponent(mx), X = Fx::out_exp(mx, E, lg);
        longlong2 v[PER][R];
#pragma unroll
        for (int p = 0; p < PER; ++p)
#pragma unroll
            for (int r = 0; r < R; ++r) v[p][r] = fx_from(x[p][r], Fx::S0, E);
        store<0, PER, R, 1>(buf, tw, v, X);
        __syncthreads();
        pass<1>(buf, tw, X);
    }
};

template <int N, int L, int PS, int T, bool INV>
struct Fft<double2, N, L, PS, T, INV> : FftShape<N, L, T, INV> {
    using Shape = FftShape<N, L, T, INV>;
    using Fx = FxPass<N, INV>;
    using Plan = FftPlan<N, INV>;
    using Shape::item;
    using Shape::NBF;
    using Shape::NBL;
    using Shape::NPASS;
    using Shape::PF;
    using Shape::PL;
    using Shape::RF;
    using Shape::RL;

    // (returns the power of two by which the values were scaled up on the way)
    template <int S, class Sync>
    __device__ static __forceinline__ int mids(longlong2* buf, const int4* __restrict__ tw, int tid, const Sync& sync) {
        if constexpr (S <= NPASS - 2) {
            constexpr int R = Plan::radix(S), Ns = Plan::ns(S), NB = N / R, PER = (NB * L + T - 1) / T;
            longlong2 v[PER][R];
#pragma unroll
            for (int p = 0; p < PER; ++p) {
                int j, line;
                if (item(p, NB, j, line, tid)) {
#pragma unroll
                    for (int r = 0; r < R; ++r) v[p][r] = buf[(j + r * NB) * PS + line];
                }
            }
            int s = 0;
            if constexpr (Fx::rescales(S)) {
                static_assert(NB * L % T == 0, "every value is set");
                s = fx_rescale<Fx, T>(v, sync);
            } else {
                sync();
            }
#pragma unroll
            for (int p = 0; p < PER; ++p) {
                int j, line;
                if (item(p, NB, j, line, tid)) {
                    Fx::template butterfly<S>(v[p], j, tw);
                    const int k = j & (Ns - 1), base = (j - k) * R + k;
#pragma unroll
                    for (int r = 0; r < R; ++r) buf[(base + r * Ns) * PS + line] = v[p][r];
                }
            }
            sync();
            return s + mids<S + 1>(buf, tw, tid, sync);
        }
        return 0;
    }
    // Block exponent of a transform from this thread's largest high word; every
    // thread of the group calls it.
    struct Scale {
        int E, X;
    };
    __device__ static __forceinline__ Scale scale_of(unsigned mx, int lg) {
        mx = fx_cta_max<T>(mx);
        const int E = fx_exponent(mx);
        return Scale{E, Fx::out_exp(mx, E, lg)};
    }
    __device__ static __forceinline__ void first_item(int p, double2 (&x)[RF], double2* dbuf, int tid, const Scale& sc) {
        longlong2* buf = reinterpret_cast<longlong2*>(dbuf);
        int j, line;
        if (item(p, NBF, j, line, tid)) {
            longlong2 v[RF];
#pragma unroll
            for (int r = 0; r < RF; ++r) v[r] = fx_from(x[r], Fx::S0, sc.E);
            dft_r<RF, INV>(v);
#pragma unroll
            for (int r = 0; r < RF; ++r) buf[(j * RF + r) * PS + line] = v[r];
        }
    }
    template <class Sync>
    __device__ static __forceinline__ void middle(double2* buf, const int4* __restrict__ tw, const int4*, int tid,
                                                  const Sync& sync, Scale& sc) {
        sync();
        sc.X -= mids<1>(reinterpret_cast<longlong2*>(buf), tw, tid, sync);
    }
    __device__ static __forceinline__ bool last_item(int p, double2 (&x)[RL], const double2* dbuf,
                                                     const int4* __restrict__ tw, const int4*, int tid, int& j,
                                                     const Scale& sc) {
        const longlong2* buf = reinterpret_cast<const longlong2*>(dbuf);
        int line;
        if (!item(p, NBL, j, line, tid)) return false;
        longlong2 v[RL];
#pragma unroll
        for (int r = 0; r < RL; ++r) v[r] = buf[(j + r * NBL) * PS + line];
        Fx::template butterfly<NPASS - 1>(v, j, tw);
#pragma unroll
        for (int r = 0; r < RL; ++r) x[r] = fx_to(v[r], sc.X);
        return true;
    }
    template <class Sync>
    __device__ static __forceinline__ void finish(const Sync& sync) { sync(); }

    template <class Sync>
    __device__ static __forceinline__ void run(double2 (&in)[PF][RF], double2 (&out)[PL][RL], double2* buf,
                                               const int4* __restrict__ tw, const int4* twl, int tid,
                                               const Sync& sync, int lg = 0) {
        unsigned mx = 0;
#pragma unroll
        for (int p = 0; p < PF; ++p) {
            int j, line;
            if (item(p, NBF, j, line, tid)) {
#pragma unroll
                for (int r = 0; r < RF; ++r) mx = max(mx, fx_hi(in[p][r]));
            }
        }
        Scale sc = scale_of(mx, lg);
        if constexpr (NPASS == 1) {
#pragma unroll
            for (int p = 0; p < PF; ++p) {
                longlong2 v[RF];
#pragma unroll
                for (int r = 0; r < RF; ++r) v[r] = fx_from(in[p][r], Fx::S0, sc.E);
                dft_r<RF, INV>(v);
#pragma unroll
                for (int r = 0; r < RF; ++r) out[p][r] = fx_to(v[r], sc.X);
            }
        } else {
#pragma unroll
            for (int p = 0; p < PF; ++p) first_item(p, in[p], buf, tid, sc);
            middle(buf, tw, twl, tid, sync, sc);
#pragma unroll
            for (int p = 0; p < PL; ++p) {
                int j;
                last_item(p, out[p], buf, tw, twl, tid, j, sc);
            }
            sync();
        }
    }
};

}  // namespace tdse
