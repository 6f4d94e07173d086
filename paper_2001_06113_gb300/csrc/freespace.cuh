// Free-space time step (Sec. 3.4, Remark highorderfs), templated on the
// transform type: FP64 (NumF64: 64-bit fixed point inside, fx.cuh) or the
// FP32-transform variant (NumF32: transforms, V u and the history sum in FP32;
// the mode state, its one-step phase p_0 and the update keep FP64 precision).
//
// One step of eq. uadamsk on the contour modes, with zeta for k and
// zeta.zeta for |k|^2 (eq. uhatxirecur):
//   W   = p_0 (u^ - i h S_1),  S_j = mu_j R_j + p_j S_{j+1}       (mode space)
//   u   = inverse(W) / (1 + i h mu_0 V)                          (grid)
//   F   = forward(V u);   u^ <- W - i h mu_0 F;   ring <- F
// The trapezoidal sub-steps of the start-up are the same with nhist = 1 and
// mu = (1/2, 1/2) (eqs. utrapzfd, uhatzfd).
//
// Transforms (fsargs.h): each axis is split into the two equispaced blocks,
// done as R interleaved M-point FFTs with folded twiddles (eq. ssfftgen), and
// the dense block of Alpert and Gauss modes, done as a direct sum.
//
// The 2R lines of M = A Bn points take two passes with the values in
// registers and one exchange through shared memory between them.  A thread
// is (line, index): grid side (line, j1) holds the points j1 + Bn j2, mode side
// (line, k2) the positions q = k2 + A k1 (mode i = s + R q of block b), so the
// grid factors, the mode factors and the whole mode update act on registers.
// Only k1 < Bn / 2 is ever used: an equispaced block fills just under half of
// its length-nu transform.  Lines are the fastest thread index: table, ring
// and state accesses of neighbouring threads are neighbouring modes.  The sum
// over the lines of a grid point (inverse) is a reduce-scatter by shuffles.
// Before, the lines made three or four round trips through shared memory per
// transform and the mode update two more, and the FP64 state update held the
// FP64 pipe 768 cycles per warp and mode (256 and about 150 integer slots now).
// Whole solves before and after: 256^2 (nu = 2048) FP64, 60 steps, 216 -> 117 ms;
// FP32 transforms, 200 steps, 110 -> 82 ms; 64^3 (nu = 256), FP32 transforms, 40
// steps, 263 -> 181 ms; 128 points (nu = 1024) FP64, 200 steps, 17.5 -> 13.5 ms.
//
// Kernels:
//   k_fs_1d   one CTA per instance: the whole 1D step;
//   k_fs_row  (2D, 3D) one CTA per mode row (k0 in 2D, (k0, k1) in 3D):
//             forward along the last axis of the row of the intermediate Z,
//             mode update and ring write (end of a step), then W of the next
//             step and its inverse along the last axis back into Z (begin of
//             a step);
//   k_fs_mid  (3D) one CTA per line (k0, j2) along axis 1: inverse from the
//             N1 modes in Z to the M1 grid values in Y, or forward back;
//   k_fs_phys (2D, 3D) one CTA per grid column (j1 in 2D, (j1, j2) in 3D):
//             inverse along axis 0 of the column of Z (3D: Y), implicit solve
//             and V u on the grid, forward along axis 0 back into the same
//             column.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

#include "cplx.cuh"
#include "device_once.h"
#include "fsargs.h"
#include "step_common.cuh"

namespace tdse {
namespace fs {

// ---------------------------------------------------------------- numbers
// NumX::C   storage type (Z, Y, ring), NumX::V register value, NumX::W table factor
struct NumF32 {
    using C = float2;
    using V = float2;
    using W = float2;
    static constexpr bool FX = false;
    template <bool CONJ, int K> static __device__ __forceinline__ V mul(V a, W w) {
        if (CONJ) w.y = -w.y;
        return cmul(a, w);
    }
    template <int LG> static __device__ __forceinline__ V div(V a) { return a; }
    static __device__ __forceinline__ V zero() { return make_float2(0.f, 0.f); }
    static __device__ __forceinline__ W load(const W* p) { return __ldg(p); }
    static __device__ __forceinline__ V shfl(V a, int o) {
        return make_float2(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o));
    }
};
struct NumF64 {
    using C = double2;
    using V = longlong2;
    using W = int4;
    static constexpr bool FX = true;
    template <bool CONJ, int K> static __device__ __forceinline__ V mul(V a, W w) { return fx_mul<CONJ, K>(a, w); }
    template <int LG> static __device__ __forceinline__ V div(V a) {       // a / 2^LG, rounded
        if (LG == 0) return a;
        constexpr long long half = LG > 0 ? 1ll << (LG > 0 ? LG - 1 : 0) : 0;
        return make_longlong2((a.x + half) >> LG, (a.y + half) >> LG);
    }
    static __device__ __forceinline__ V zero() { return make_longlong2(0, 0); }
    static __device__ __forceinline__ W load(const W* p) { return __ldg(p); }
    static __device__ __forceinline__ V shfl(V a, int o) {
        return make_longlong2(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o));
    }
};

// Tables of an axis.
template <class N> struct Tab;
template <> struct Tab<NumF64> {
    static __device__ __forceinline__ const int4* preI(const FsAxis& a) { return a.preI; }
    static __device__ __forceinline__ const int4* postI(const FsAxis& a) { return a.postI; }
    static __device__ __forceinline__ const int4* preF(const FsAxis& a) { return a.preF; }
    static __device__ __forceinline__ const int4* postF(const FsAxis& a) { return a.postF; }
    static __device__ __forceinline__ const int4* Gd(const FsAxis& a) { return a.Gd; }
    static __device__ __forceinline__ const int4* Fd(const FsAxis& a) { return a.Fd; }
    static __device__ __forceinline__ const int4* tw(const FsAxis& a) { return a.tw; }
    static __device__ __forceinline__ const int4* Lf(const FsAxis& a) { return a.Lf; }
    static __device__ __forceinline__ const int4* Li(const FsAxis& a) { return a.Li; }
    static __device__ __forceinline__ const double* Tc(const FsAxis& a) { return a.Tc; }
    static __device__ __forceinline__ const double2* TcW(const FsAxis& a) { return a.TcW; }
};
template <> struct Tab<NumF32> {
    static __device__ __forceinline__ const float2* preI(const FsAxis& a) { return a.preI_f; }
    static __device__ __forceinline__ const float2* postI(const FsAxis& a) { return a.postI_f; }
    static __device__ __forceinline__ const float2* preF(const FsAxis& a) { return a.preF_f; }
    static __device__ __forceinline__ const float2* postF(const FsAxis& a) { return a.postF_f; }
    static __device__ __forceinline__ const float2* Gd(const FsAxis& a) { return a.Gd_f; }
    static __device__ __forceinline__ const float2* Fd(const FsAxis& a) { return a.Fd_f; }
    static __device__ __forceinline__ const float2* tw(const FsAxis& a) { return a.tw_f; }
    static __device__ __forceinline__ const float2* Lf(const FsAxis& a) { return a.Lf_f; }
    static __device__ __forceinline__ const float2* Li(const FsAxis& a) { return a.Li_f; }
    static __device__ __forceinline__ const float* Tc(const FsAxis& a) { return a.Tc_f; }
    static __device__ __forceinline__ const float2* TcW(const FsAxis& a) { return a.TcW_f; }
};

// ---------------------------------------------------------------- short DFTs
// HALF: inputs n/2 .. n-1 are zero.  Result q at v[at(q)].
template <bool INV, class V> __device__ __forceinline__ void dft4_half(V& a0, V& a1, V& a2, V& a3) {
    const V x = a0, y = a1, r = rot90<INV>(a1);
    a0 = x + y;
    a2 = x - y;
    a1 = x + r;
    a3 = x - r;
}
template <bool INV, bool HALF, class V> __device__ __forceinline__ void dft4_any(V& a0, V& a1, V& a2, V& a3) {
    if (HALF) dft4_half<INV>(a0, a1, a2, a3);
    else dft4<INV>(a0, a1, a2, a3);
}
// e^{-+ i pi k / 8}, k odd
template <bool INV, int KK> __device__ __forceinline__ float2 rot16(float2 v) {
    constexpr float c = 0.92387953251128675613f, s = 0.38268343236508977173f;
    constexpr float wc = KK == 1 ? c : (KK == 3 ? s : -c), ws = KK == 1 ? -s : (KK == 3 ? -c : s);
    return cmul(v, make_float2(wc, INV ? -ws : ws));
}
template <bool INV, int KK> __device__ __forceinline__ longlong2 rot16(longlong2 v) {
    const int ch = 496004047, cl = 848119337, sh = 205451603, sl = 1465168233;      // cos, sin (pi / 8) in limbs
    const int4 w = KK == 1 ? make_int4(ch, cl, -sh, -sl) : (KK == 3 ? make_int4(sh, sl, -ch, -cl) : make_int4(-ch, -cl, sh, sl));
    return fx_mul<INV, 3>(v, w);
}
template <int N, bool INV, bool HALF> struct Dft;
template <bool INV, bool HALF> struct Dft<4, INV, HALF> {
    static constexpr int at(int q) { return q; }
    template <class V> static __device__ __forceinline__ void run(V* v) { dft4_any<INV, HALF>(v[0], v[1], v[2], v[3]); }
};
template <bool INV, bool HALF> struct Dft<8, INV, HALF> {
    static constexpr int at(int q) { return q; }
    template <class V> static __device__ __forceinline__ void run(V* v) {
        V e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
        dft4_any<INV, HALF>(e0, e1, e2, e3);
        dft4_any<INV, HALF>(o0, o1, o2, o3);
        o1 = rot45<INV>(o1);
        o2 = rot90<INV>(o2);
        o3 = rot90<INV>(rot45<INV>(o3));
        v[0] = e0 + o0; v[4] = e0 - o0;
        v[1] = e1 + o1; v[5] = e1 - o1;
        v[2] = e2 + o2; v[6] = e2 - o2;
        v[3] = e3 + o3; v[7] = e3 - o3;
    }
};
template <bool INV, bool HALF> struct Dft<16, INV, HALF> {
    static constexpr int at(int q) { return 4 * (q & 3) + (q >> 2); }
    template <class V> static __device__ __forceinline__ void run(V* v) {
#pragma unroll
        for (int c = 0; c < 4; ++c) dft4_any<INV, HALF>(v[c], v[c + 4], v[c + 8], v[c + 12]);
        v[5] = rot16<INV, 1>(v[5]);
        v[6] = rot45<INV>(v[6]);
        v[7] = rot16<INV, 3>(v[7]);
        v[9] = rot45<INV>(v[9]);
        v[10] = rot90<INV>(v[10]);
        v[11] = rot90<INV>(rot45<INV>(v[11]));
        v[13] = rot16<INV, 3>(v[13]);
        v[14] = rot90<INV>(rot45<INV>(v[14]));
        v[15] = rot16<INV, 9>(v[15]);
#pragma unroll
        for (int k = 0; k < 4; ++k) dft4<INV>(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
    }
};

// ---------------------------------------------------------------- geometry
// Grids of M > 256 points use transforms of M / 2 points on twice the lines
// (e^{2 pi i (s + R' q) j / nu} has period M / 2 in j up to the folded factor
// e^{2 pi i s j / nu}): each transform point serves FOLD grid points.
template <int M_, int R_> struct Geo {
    static constexpr int M = M_;
    static constexpr int FOLD = M > 256 ? 2 : 1;
    static constexpr int MF = M / FOLD;              // transform length
    static constexpr int R = R_ * FOLD;              // lines per block
    static constexpr int L = 2 * R;
    static constexpr int A = MF >= 128 ? 16 : (MF == 64 ? 8 : 4);
    static constexpr int B = MF / A;
    static constexpr int NV = B / 2;                 // equispaced modes per mode-side thread
    static constexpr int T = L * (A > B ? A : B);
    static constexpr int FPT = (M + T - 1) / T;      // grid points per thread
    static constexpr int PB = B * L + (L == 8 ? 8 : 0);   // exchange row (8 lines: padded against bank conflicts)
    static constexpr int XBUF = A * PB;
    static constexpr int ROWS = FS_MAX_ND + FS_MAX_NT;
    static constexpr int LA = ilog2(A), LB = ilog2(B), LR = ilog2(R), LF = ilog2(FOLD), LM = ilog2(M);
};
// Resident CTAs: 2 of 256 threads for the fixed-point kernels (up to 128
// registers), FS_MINB32 for the FP32 ones (256^2, per step: 3, 4, 5, 6 CTAs 317,
// 294, 289, 329 us).
#ifndef FS_MINB32
#define FS_MINB32 5
#endif
template <class N, class G> constexpr int min_blocks() {
    const int t = N::FX ? 512 : 256 * FS_MINB32;
    return t / G::T < 1 ? 1 : (t / G::T > 16 ? 16 : t / G::T);
}

template <class N, class G> struct Smem {
    typename N::V x[G::XBUF];          // exchange between the two sides
    typename N::V f[N::FX ? 3 : 2][G::M];   // grid values: see put_grid and inverse
    typename N::C d[G::ROWS];          // dense modes, then the interpolant's terms
    longlong2 dl[N::FX ? G::ROWS : 1]; // the same in fixed point (inverse)
    int4 c[FS_MAX_HIST + 1];           // row phases: c[0] p_0's row factor; F64: c_j; F32: c_j as floats (x, y)
    unsigned red[5][32];
};

template <int T> __device__ __forceinline__ unsigned cta_max(unsigned v, unsigned* red) {
    v = __reduce_max_sync(0xffffffffu, v);
    if constexpr (T > 32) {
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
        __syncthreads();
        v = __reduce_max_sync(0xffffffffu, red[(threadIdx.x & 31) % (T / 32)]);
    }
    return v;
}

template <class N, int M, int R_>
struct Line {
    using G = Geo<M, R_>;
    using V = typename N::V;
    using C = typename N::C;
    using T = Tab<N>;
    using Sm = Smem<N, G>;
    static constexpr int R = G::R, L = G::L, A = G::A, B = G::B, NV = G::NV;

    // mode of position k1 of this thread: -1 where it holds none
    __device__ static __forceinline__ int mode(int k1, const FsAxis& ax) {
        const int line = threadIdx.x % L, k2 = threadIdx.x / L, b = line / R, s = line % R;
        const int i = s + R * (k2 + A * k1);
        if (k2 >= A || i >= ax.NE) return -1;
        return b ? ax.NE + ax.ND + i : i;
    }
    __device__ static __forceinline__ int index(int m, const FsAxis& ax) { return m < ax.NE ? m : m - ax.ND; }   // [2][NE]

    // Exponents of a fixed-point forward transform's inputs: the two equispaced
    // blocks and the dense rows (FX_NAN: a NaN or an infinity).
    struct GridExp {
        int e[3];
    };
    // Grid values f[p] of points tid + p T -> shared memory.  F64: the factors of
    // a block have moduli 2^x_j (times 1/2..1) that span e^{+-H}; a point is held
    // relative to the largest |f_j| 2^x_j of its block, as an FP64 sum would
    // weigh it, and the factors are scaled to modulus 1.  Ends with a barrier.
    __device__ static __forceinline__ GridExp put_grid(const C (&f)[G::FPT], Sm& sm, const FsAxis& ax) {
        GridExp g{};
        if constexpr (N::FX) {
            unsigned mx[3] = {0, 0, 0};
#pragma unroll
            for (int p = 0; p < G::FPT; ++p) {
                const int j = threadIdx.x + p * G::T;
                if (G::M % G::T != 0 && j >= M) continue;
                const unsigned h = fx_hi(f[p]);
                const int e = fx_exponent(h);
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    mx[c] = max(mx[c], h >= 0x7ff00000u ? 0xffffffffu : (unsigned)(e + __ldg(&ax.xj[c * M + j]) + 16384));
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                mx[c] = __reduce_max_sync(0xffffffffu, mx[c]);
                if ((threadIdx.x & 31) == 0) sm.red[2 + c][threadIdx.x >> 5] = mx[c];
            }
            __syncthreads();
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const unsigned v = __reduce_max_sync(0xffffffffu, sm.red[2 + c][(threadIdx.x & 31) % (G::T / 32)]);
                g.e[c] = v == 0xffffffffu ? FX_NAN : (int)v - 16384;
            }
        }
#pragma unroll
        for (int p = 0; p < G::FPT; ++p) {
            const int j = threadIdx.x + p * G::T;
            if (G::M % G::T != 0 && j >= M) continue;
            if constexpr (N::FX) {
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    sm.f[c][j] = fx_from(f[p], 61, g.e[c] >= FX_NAN ? 2046 : g.e[c] - __ldg(&ax.xj[c * M + j]));
            } else {
                sm.f[0][j] = f[p];
            }
        }
        __syncthreads();
        return g;
    }

    // This thread's own slot of sm.x for its position k1 (no other thread touches
    // it between the exchanges): results of forward, inputs of inverse.
    __device__ static __forceinline__ V* slot(Sm& sm, int k1) {
        return &sm.x[(threadIdx.x / L) * G::PB + k1 * L + threadIdx.x % L];
    }

    // Forward transform of the grid values in sm.f (put_grid).  On return *slot(k1)
    // is the equispaced mode `mode(k1)` (F64: times 2^-xe) and sm.d the dense
    // modes 0 .. ND-1, complete after the call's last barrier.
    __device__ static __forceinline__ void forward(Sm& sm, const FsAxis& ax, const GridExp& ge, int& xe) {
        constexpr int KF = 4 - G::LA - G::LF, KB = 3 - G::LB, KD = 4 - G::LM;
        const int line = threadIdx.x % L, idx = threadIdx.x / L, b = line / R, s = line % R;
        if (idx < B) {
            V x[A];
            const V* f = sm.f[N::FX ? b : 0];
            const typename N::W* pre = T::preF(ax) + (size_t)b * M * R + s;
#pragma unroll
            for (int j2 = 0; j2 < A; ++j2) {
                const int j = idx + B * j2;
                x[j2] = N::template mul<false, KF>(f[j], N::load(pre + (size_t)j * R));
                if constexpr (G::FOLD == 2)
                    x[j2] = x[j2] + N::template mul<false, KF>(f[j + G::MF], N::load(pre + (size_t)(j + G::MF) * R));
            }
            Dft<A, false, false>::run(x);
            const typename N::W* tw = T::tw(ax);
#pragma unroll
            for (int k2 = 0; k2 < A; ++k2) {
                V y = x[Dft<A, false, false>::at(k2)];
                if (k2 == 0) y = N::template div<G::LB>(y);
                else y = N::template mul<false, KB>(y, N::load(tw + idx * k2));
                sm.x[k2 * G::PB + idx * L + line] = y;
            }
        }
        // dense rows by warps: direct sums (the C rows are not kept when they go
        // through the interpolant), then the NT interpolant rows
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        const bool cheb = ax.NT > 0;
        const int nrow = ax.ND + (cheb ? ax.NT : 0);
        const int xd = ge.e[2] - 1083 + 3 - KD;
        const V* fd = sm.f[N::FX ? 2 : 0];
        for (int r0 = 4 * warp; r0 < nrow; r0 += G::T / 8) {      // four rows at a time
            V acc[4];
            const typename N::W* row[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int rr = min(r0 + q, nrow - 1);
                acc[q] = N::zero();
                row[q] = rr >= ax.ND ? T::Lf(ax) + (rr - ax.ND) * M : T::Fd(ax) + rr * M;
            }
#pragma unroll(N::FX ? 1 : 2)
            for (int j = lane; j < M; j += 32) {
                const V x = fd[j];
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[q] = acc[q] + N::template mul<false, KD>(x, N::load(row[q] + j));
            }
            // sums over the lanes: after two exchanges a lane holds a part of one row
            const bool h16 = lane & 16, h8 = lane & 8;
#pragma unroll
            for (int q = 0; q < 2; ++q) acc[q] = (h16 ? acc[q + 2] : acc[q]) + N::shfl(h16 ? acc[q] : acc[q + 2], 16);
            acc[0] = (h8 ? acc[1] : acc[0]) + N::shfl(h8 ? acc[0] : acc[1], 8);
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) acc[0] = acc[0] + N::shfl(acc[0], o);
            const int rr = r0 + (h16 ? 2 : 0) + (h8 ? 1 : 0);
            if ((lane & 7) == 0 && rr < nrow && !(cheb && rr >= ax.p && rr < ax.p + ax.NC)) {
                C r;
                if constexpr (N::FX) r = fx_to(acc[0], ge.e[2] >= FX_NAN ? FX_NAN : xd);
                else r = acc[0];
                sm.d[rr >= ax.ND ? FS_MAX_ND + rr - ax.ND : rr] = r;
            }
        }
        __syncthreads();
        if (cheb) {   // C rows: f^_k = sum_l T_l(tau_k / H) g_l
            for (int k = threadIdx.x; k < ax.NC; k += G::T) {
                const auto* tc = T::Tc(ax) + (size_t)k * ax.NT;
                C acc = czero<C>();
                for (int l = 0; l < ax.NT; ++l) acc = acc + cscale(sm.d[FS_MAX_ND + l], __ldg(&tc[l]));
                sm.d[ax.p + k] = acc;
            }
            __syncthreads();
        }
        if (idx < A) {
            V x[B];
#pragma unroll
            for (int j1 = 0; j1 < B; ++j1) x[j1] = sm.x[idx * G::PB + j1 * L + line];
            Dft<B, false, false>::run(x);
#pragma unroll
            for (int k1 = 0; k1 < NV; ++k1) {
                const int m = mode(k1, ax);
                if (m >= 0)
                    *slot(sm, k1) = N::template mul<false, 3>(x[Dft<B, false, false>::at(k1)], N::load(T::postF(ax) + index(m, ax)));
            }
        }
        xe = ge.e[b] >= FX_NAN ? FX_NAN : ge.e[b] - 1083 + 3 - KF + G::LB;
    }

    // Inverse transform of the modes in *slot(k1) (equispaced, as C; mx: the
    // largest fx_hi of this thread's) and sm.d[0..ND) (dense): y[p] = grid value
    // of point tid + p T.  Begins with a barrier (sm.d written, sm.f free).
    __device__ static __forceinline__ void inverse(Sm& sm, unsigned mx, C (&y)[G::FPT], const FsAxis& ax) {
        constexpr int KI = 5 - G::LB, KA = 3 - G::LA, KL = 3 - G::LR;
        const int line = threadIdx.x % L, idx = threadIdx.x / L, b = line / R, s = line % R;
        int E = 0, Ed = 0;
        if constexpr (N::FX) {
            mx = cta_max<G::T>(mx, sm.red[1]);
            E = mx >= 0x7ff00000u ? FX_NAN : fx_exponent(mx);
        } else {
            __syncthreads();
        }
        const bool cheb = ax.NT > 0;
        if (cheb) {   // h_l = sum_k T_l(tau_k / H) (w_k / 2pi) f^_k
            for (int l = threadIdx.x; l < ax.NT; l += G::T) {
                const C* tw = T::TcW(ax) + (size_t)l * ax.NC;
                C acc = czero<C>();
                for (int k = 0; k < ax.NC; ++k) acc = acc + cmul(__ldg(&tw[k]), sm.d[ax.p + k]);
                sm.d[FS_MAX_ND + l] = acc;
            }
            __syncthreads();
        }
        if constexpr (N::FX) {   // block exponent of the dense rows (every warp for itself), limbs of its share
            unsigned mx = 0;
            for (int r = threadIdx.x & 31; r < ax.ND; r += 32) mx = max(mx, fx_hi(sm.d[r]));
            for (int r = threadIdx.x & 31; r < (cheb ? ax.NT : 0); r += 32) mx = max(mx, fx_hi(sm.d[FS_MAX_ND + r]));
            mx = __reduce_max_sync(0xffffffffu, mx);
            Ed = mx >= 0x7ff00000u ? FX_NAN : fx_exponent(mx);
            for (int r = threadIdx.x; r < G::ROWS; r += G::T)
                if (r < ax.ND || (cheb && r >= FS_MAX_ND && r < FS_MAX_ND + ax.NT))
                    sm.dl[r] = fx_from(sm.d[r], 55, Ed >= FX_NAN ? 2046 : Ed);
        }
        if (idx < A) {
            V x[B];
#pragma unroll
            for (int k1 = 0; k1 < B; ++k1) x[k1] = N::zero();
#pragma unroll
            for (int k1 = 0; k1 < NV; ++k1) {
                const int m = mode(k1, ax);
                if (m >= 0) {
                    V wv;
                    if constexpr (N::FX) wv = fx_from(*reinterpret_cast<const C*>(slot(sm, k1)), 61, E >= FX_NAN ? 2046 : E);
                    else wv = *slot(sm, k1);
                    x[k1] = N::template mul<false, KI>(wv, N::load(T::preI(ax) + index(m, ax)));
                }
            }
            Dft<B, true, true>::run(x);
            const typename N::W* tw = T::tw(ax);
#pragma unroll
            for (int j1 = 0; j1 < B; ++j1) {
                V z = x[Dft<B, true, true>::at(j1)];
                if (j1 == 0) z = N::template div<G::LA>(z);
                else z = N::template mul<true, KA>(z, N::load(tw + idx * j1));
                sm.x[idx * G::PB + j1 * L + line] = z;
            }
        }
        __syncthreads();
        // (every thread of a warp takes part in the shuffles: T is a multiple of B L and of 32)
        if (idx < B) {
            V x[A];
#pragma unroll
            for (int k2 = 0; k2 < A; ++k2) x[k2] = sm.x[k2 * G::PB + idx * L + line];
            Dft<A, true, false>::run(x);
            const typename N::W* post = T::postI(ax) + (size_t)b * M * R + s;
#pragma unroll
            for (int t = 0; t < G::FOLD; ++t) {
                V z[A];
#pragma unroll
                for (int j2 = 0; j2 < A; ++j2)
                    z[j2] = N::template mul<false, KL>(x[Dft<A, true, false>::at(j2)],
                                                       N::load(post + (size_t)(idx + B * j2 + t * G::MF) * R));
                int j2 = 0;
                reduce<A, R / 2>(z, line, j2);
                constexpr int LEFT = A > R ? A / R : 1;          // sums this thread ends with: points j2 .. j2 + LEFT - 1
                constexpr int DUP = R > A ? R / A : 1;           // threads that hold the same sum
                if (line % DUP == 0) {
#pragma unroll
                    for (int i = 0; i < LEFT; ++i) sm.f[b][idx + B * (j2 + i) + t * G::MF] = z[i];
                }
            }
        }
        __syncthreads();
        const int xe = E - 1083 + ax.xI + 3 - KI + G::LA + G::LR, xd = Ed - 1022 - 55;
        const typename N::W* gd = T::Gd(ax);
        const typename N::W* li = T::Li(ax);
#pragma unroll
        for (int p = 0; p < G::FPT; ++p) {
            const int j = threadIdx.x + p * G::T;
            y[p] = czero<C>();
            if (G::M % G::T != 0 && j >= M) continue;
            V acc = N::zero();
            auto rows = [&](const typename N::W* t, int first, int last, int at) {
#pragma unroll 4
                for (int r = first; r < last; ++r) {
                    if constexpr (N::FX) acc = acc + fx_mul<false, 3>(sm.dl[at + r], N::load(t + (size_t)r * M + j));
                    else acc = acc + cmul(N::load(t + (size_t)r * M + j), sm.d[at + r]);
                }
            };
            if (!cheb) {
                rows(gd, 0, ax.ND, 0);
            } else {   // Alpert rows directly, the C rows as sum_l rho_l(x_j) h_l
                rows(gd, 0, ax.p, 0);
                rows(gd, ax.p + ax.NC, ax.ND, 0);
                rows(li, 0, ax.NT, FS_MAX_ND);
            }
            if constexpr (N::FX) {
                auto at = [&](V v, int c, int x, bool bad) { return fx_to(v, bad ? FX_NAN : x + __ldg(&ax.xj[c * M + j])); };
                y[p] = at(sm.f[0][j], 3, xe, E >= FX_NAN) + at(sm.f[1][j], 4, xe, E >= FX_NAN) + at(acc, 5, xd, Ed >= FX_NAN);
            } else {
                y[p] = sm.f[0][j] + sm.f[1][j] + acc;
            }
        }
    }

    // Sum of z[0..n) over the R lines of a block at a grid index, scattered: halves while a
    // thread has more than one sum, then whole sums.
    template <int n, int o>
    __device__ static __forceinline__ void reduce(V* z, int line, int& at) {
        if constexpr (o >= 1) {
            if constexpr (n > 1) {
                const bool up = line & o;
#pragma unroll
                for (int i = 0; i < n / 2; ++i) {
                    const V send = up ? z[i] : z[i + n / 2], keep = up ? z[i + n / 2] : z[i];
                    z[i] = keep + N::shfl(send, o);
                }
                if (up) at += n / 2;
                reduce<n / 2, o / 2>(z, line, at);
            } else {
                z[0] = z[0] + N::shfl(z[0], o);
                reduce<1, o / 2>(z, line, at);
            }
        }
    }
};

// ---------------------------------------------------------------- mode update
// One-step phases are factors in units of 2^-(60 - g) (|p| < 2^(1 + g); g of the
// instance, 0 unless its field moves the contour phases by more than a factor
// of 2 over the history, see fs_api.cpp); from g = FS_WIDE on they and the history
// sum are FP64 (WIDE below).  A CTA takes one form or the other for the whole of
// its modes, the FP64 one in functions of their own: a branch per mode cost the
// fixed-point form 0.4 to 2.8 %.
__device__ __forceinline__ longlong2 pmul(longlong2 v, int4 p, int g) {
    longlong2 r = fx_mul<false, 4>(v, p);
    if (g) r = make_longlong2((long long)((unsigned long long)r.x << g), (long long)((unsigned long long)r.y << g));
    return r;
}
__device__ __forceinline__ double2 wide_phase(int4 p) {
    return make_double2(__hiloint2double(p.y, p.x), __hiloint2double(p.w, p.z));
}
__device__ __forceinline__ int4 wide_bits(double2 v) {
    return make_int4(__double2loint(v.x), __double2hiint(v.x), __double2loint(v.y), __double2hiint(v.y));
}
template <bool WIDE> __device__ __forceinline__ int4 phase_one(int g) {
    return WIDE ? wide_bits(make_double2(1.0, 0.0)) : make_int4(1 << (28 - g), 0, 0, 0);
}
template <bool WIDE> __device__ __forceinline__ int4 phase_mul(int4 a, int4 b, int g) {
    if constexpr (WIDE) return wide_bits(cmul(wide_phase(a), wide_phase(b)));
    else return fx_as_factor(pmul(fx_value(a), b, g));
}

__device__ __forceinline__ float2 to_c(double2 v, float2) { return fx_to_float(v); }
__device__ __forceinline__ double2 to_c(double2 v, double2) { return v; }

__device__ __forceinline__ double2 widen(float2 x) { return fx_widen(x); }
__device__ __forceinline__ double2 widen(double2 x) { return x; }
template <class C> constexpr int widens() { return std::is_same<C, float2>::value ? 1 : 0; }     // index of up_h, up_hmu0
// v * (-i c) added to u
__device__ __forceinline__ double2 add_minus_i(double2 u, double c, double2 v) {
    return make_double2(fma(c, v.y, u.x), fma(-c, v.x, u.y));
}

// c R + b S with one rounding per fused multiply-add (complex).
__device__ __forceinline__ float2 cmul_add2(float2 c, float2 R, float2 b, float2 S) {
    return make_float2(fmaf(c.x, R.x, fmaf(-c.y, R.y, fmaf(b.x, S.x, -b.y * S.y))),
                       fmaf(c.x, R.y, fmaf(c.y, R.x, fmaf(b.x, S.y, b.y * S.x))));
}

// Where a row's modes live: lag[j - 1] the ring slot of lag j, pc[j] the phases
// b_j of its lags, p0 those of the step, all at mode 0 of the row.
template <class N> struct PhaseTab;
template <class N> struct RowPtr {
    using C = typename N::C;
    const double2* src;
    double2* uh;
    C* out;
    const C* lag[FS_MAX_HIST];
    const typename PhaseTab<N>::type* pc[FS_MAX_HIST];
    const int4* p0;
    bool first_is_new;          // lag 1 is the value this launch computes
};

// History sum of eq. uadamsk in Horner form with separable phases p_i = a_i b_i
// (a_i of the row, b_i of the mode; 1D: a_i = 1):  S_j = c_j R_j + b_j S_{j+1},
// c_j = mu_j a_1 .. a_{j-1}, so that S_1 = sum_j mu_j p_1 .. p_{j-1} R_j.
// F32: in FP32; F64: in fixed point, the R_j sharing an exponent (WIDE: in FP64).
template <bool WIDE>
__device__ __forceinline__ float2 history(const FsArgs& a, int g, const int4* c, const float2 (&r)[FS_MAX_HIST],
                                          const float2* const (&pc)[FS_MAX_HIST], int m) {
    float2 S = make_float2(0.f, 0.f);
#pragma unroll
    for (int j = FS_MAX_HIST; j >= 1; --j) {
        if (j <= a.nhist) {
            const int2 w = *reinterpret_cast<const int2*>(&c[j]);
            const float2 cj = make_float2(__int_as_float(w.x), __int_as_float(w.y));
            if (j < FS_MAX_HIST && j < a.nhist) S = cmul_add2(cj, r[j - 1], __ldg(pc[j] + m), S);
            else S = cmul(cj, r[j - 1]);
        }
    }
    return S;
}
template <bool WIDE>
__device__ __forceinline__ double2 history(const FsArgs& a, int g, const int4* c, const double2 (&r)[FS_MAX_HIST],
                                           const int4* const (&pc)[FS_MAX_HIST], int m) {
    if constexpr (WIDE) {
        double2 S = make_double2(0.0, 0.0);
#pragma unroll
        for (int j = FS_MAX_HIST; j >= 1; --j) {
            if (j <= a.nhist) {
                if (j < FS_MAX_HIST && j < a.nhist) S = cmul(S, wide_phase(__ldg(pc[j] + m)));
                S = S + cmul(wide_phase(c[j]), r[j - 1]);
            }
        }
        return S;
    } else {
    unsigned mr = 0;
#pragma unroll
    for (int j = 0; j < FS_MAX_HIST; ++j) mr = max(mr, fx_hi(r[j]));
    const int E = fx_exponent(mr), S0 = 58 - g;      // |S| < 4.4 2^(S0 + 1.5 + g) < 2^62
    longlong2 S = make_longlong2(0, 0);
#pragma unroll
    for (int j = FS_MAX_HIST; j >= 1; --j) {
        if (j <= a.nhist) {
            if (j < FS_MAX_HIST && j < a.nhist) S = pmul(S, __ldg(pc[j] + m), g);
            S = S + pmul(fx_from(r[j - 1], S0, E), c[j], g);
        }
    }
    return fx_to(S, mr >= 0x7ff00000u ? FX_NAN : E - 1022 - S0);
    }
}

template <> struct PhaseTab<NumF32> {
    using type = float2;
    static __device__ __forceinline__ const float2* get(const FsAxis& ax) { return ax.P_f; }
};
template <> struct PhaseTab<NumF64> {
    using type = int4;
    static __device__ __forceinline__ const int4* get(const FsAxis& ax) { return ax.P; }
};

// Row factors of a begin, by the last warp of the CTA into sm.c (the caller's
// next barrier publishes them): c[0] = a_0, c[j] = mu_j a_1 .. a_{j-1}; phase(i)
// is the row's factor a_i.  Lane i holds a_i, a scan over the lanes the products.
template <class N, bool WIDE, class Sm, class Ph>
__device__ __forceinline__ void row_factors(const FsArgs& a, int g, Sm& sm, int T, Ph phase) {
    const int lane = (int)threadIdx.x - (T - 32);
    if (lane < 0) return;
    const int4 one = phase_one<WIDE>(g);
    const int nh = min(a.nhist, FS_MAX_HIST);
    int4 A = lane == 0 || lane < nh ? phase(lane) : one;
    if (lane == 0) {
        sm.c[0] = A;
        A = one;
    }
#pragma unroll 1
    for (int o = 1; o < 8; o <<= 1) {
        const int4 B = make_int4(__shfl_up_sync(0xffffffffu, A.x, o), __shfl_up_sync(0xffffffffu, A.y, o),
                                 __shfl_up_sync(0xffffffffu, A.z, o), __shfl_up_sync(0xffffffffu, A.w, o));
        const int4 P = phase_mul<WIDE>(A, B, g);
        if (lane >= o) A = P;
    }
    const int j = lane + 1;                            // A = a_1 .. a_{j-1}
    if (j > nh) return;
    const longlong2 v = fx_value(A);
    if constexpr (N::FX) {
        if constexpr (WIDE) sm.c[j] = wide_bits(cscale(wide_phase(A), a.mu[j]));
        else sm.c[j] = fx_as_factor(make_longlong2(fx_mul_real<4>(v.x, a.mu_w[j]), fx_mul_real<4>(v.y, a.mu_w[j])));
    } else {
        double2 d;
        if constexpr (WIDE) d = wide_phase(A);
        else d = fx_to(v, g - 60);
        sm.c[j] = make_int4(__float_as_int((float)(a.mu[j] * d.x)), __float_as_int((float)(a.mu[j] * d.y)), 0, 0);
    }
}

template <class N>
__device__ __forceinline__ RowPtr<N> row_ptr(const FsArgs& a, bool end, const double2* src, double2* uh, typename N::C* ring, size_t slot_stride,
                                             const int4* P, const typename PhaseTab<N>::type* Pc, int Nm) {
    RowPtr<N> p;
    p.src = src;
    p.uh = uh;
    p.out = ring + (size_t)(a.out_slot < 0 ? 0 : a.out_slot) * slot_stride;      // (not written by a begin alone)
#pragma unroll
    for (int j = 0; j < FS_MAX_HIST; ++j) {
        const int i = j < a.nhist ? j : 0;
        p.lag[j] = ring + (size_t)a.hist_slot[i] * slot_stride;
        p.pc[j] = Pc + (size_t)a.interval[i] * Nm;
    }
    p.p0 = P + (size_t)a.interval[0] * Nm;
    p.first_is_new = end && a.nhist > 0 && a.hist_slot[0] == a.out_slot;
    return p;
}

// Mode m of a row: end of a step (state, ring slot; F the new (Vu)^) and/or
// begin of the next (W, returned; also left in the state).  The sums u^ - i h
// mu_0 F and u^ - i h S are FP64 fused multiply-adds (4 of them: their 256
// cycles of the FP64 pipe run beside the integer work of other warps), the
// phase product p_0 X, 8 more in FP64, is done in fixed point.
template <class N, bool WIDE>
__device__ __forceinline__ double2 update_mode(const FsArgs& a, int g, const int4* c, bool end, bool begin, int m,
                                               typename N::C F, const RowPtr<N>& p) {
    using C = typename N::C;
    double2 u = p.src[m];
    C r[FS_MAX_HIST];
    int4 b0 = make_int4(0, 0, 0, 0);
    if (begin) {
#pragma unroll
        for (int j = 0; j < FS_MAX_HIST; ++j)
            r[j] = j < a.nhist && !(j == 0 && p.first_is_new) ? p.lag[j][m] : czero<C>();
        b0 = __ldg(p.p0 + m);
    }
    if (end) {
        p.out[m] = F;
        u = add_minus_i(u, a.up_hmu0[widens<C>()], widen(F));
        if (!begin) {
            p.uh[m] = u;
            return u;
        }
        if (p.first_is_new) r[0] = F;
    }
    const double2 X = add_minus_i(u, a.up_h[widens<C>()], widen(history<WIDE>(a, g, c, r, p.pc, m)));
    double2 W;
    if constexpr (!WIDE) {
        const unsigned mx = fx_hi(X);
        const int E = fx_exponent(mx);
        const longlong2 v = pmul(pmul(fx_from(X, 59, E), c[0], g), b0, g);
        W = fx_to(v, mx >= 0x7ff00000u ? FX_NAN : E - 1022 - 59);
    } else {
        W = cmul(cmul(X, wide_phase(c[0])), wide_phase(b0));
    }
    p.uh[m] = W;
    return W;
}

// u = y / (1 + i c)
__device__ __forceinline__ float2 implicit_solve(float2 y, float c) {
    const float den = 1.f + c * c;
    return make_float2((y.x + c * y.y) / den, (y.y - c * y.x) / den);
}
__device__ __forceinline__ double2 implicit_solve(double2 y, double c) {
    const double q = recip_any(fma(c, c, 1.0));
    return make_double2(fma(c, y.y, y.x) * q, fma(-c, y.x, y.y) * q);
}

template <class C>
__device__ __forceinline__ void store_fwd(const FsArgs& a, size_t idx, C F) {
    if (a.fdst_ring) reinterpret_cast<C*>(a.fdst)[idx] = F;
    else a.fdst[idx] = cvt<double2>(F);
}
template <class N>
__device__ __forceinline__ typename N::C mode_value(typename N::V v, int xe) {
    if constexpr (N::FX) return fx_to(v, xe);
    else return v;
}

// f(m, F, W) for every mode m of this thread, equispaced and dense: F its
// forward result (where have_F), W where its input of the inverse transform
// goes.  One rolled loop: the mode update is the kernel's largest piece of code.
// (Loads issued one mode ahead were slower: 307 to 356 us, for 3 to 5 CTAs.)
template <class N, class Ln, class Fn>
__device__ __forceinline__ void each_mode(const FsAxis& ax, typename Ln::Sm& sm, bool have_F, int xe, Fn f) {
    using C = typename N::C;
    const int extra = (ax.ND + Ln::G::T - 1) / Ln::G::T;
    const int line = threadIdx.x % Ln::L, k2 = threadIdx.x / Ln::L, b = line / Ln::R;
    int i = k2 < Ln::A ? line % Ln::R + Ln::R * k2 : ax.NE;               // position in the block, + R A per k1
    int d = (int)threadIdx.x - Ln::NV * Ln::G::T;
    typename N::V* at = Ln::slot(sm, 0);
    const int m0 = b ? ax.NE + ax.ND : 0;
#pragma unroll 1
    for (int k = 0; k < Ln::NV + extra; ++k, i += Ln::R * Ln::A, d += Ln::G::T, at += Ln::L) {
        const bool dense = k >= Ln::NV;
        if (dense ? d >= ax.ND : i >= ax.NE) continue;
        C* w = dense ? &sm.d[d] : reinterpret_cast<C*>(at);
        C F = czero<C>();
        if (have_F) F = dense ? *w : mode_value<N>(*at, xe);
        f(dense ? ax.NE + d : m0 + i, F, w);
    }
}

// What locates the modes of a row (row_ptr's arguments).
template <class N> struct RowArgs {
    const double2* src;
    double2* uh;
    typename N::C* ring;
    size_t slot_stride;
    const int4* P;
    const typename PhaseTab<N>::type* Pc;
};

// Every mode of this thread through update_mode (end and / or begin); returns
// the largest fx_hi of its inputs of the inverse transform (FP64).
template <class N, class Ln, bool WIDE>
__device__ __forceinline__ unsigned update_modes(const FsArgs& a, const FsAxis& ax, typename Ln::Sm& sm, int g, bool end,
                                                 bool begin, int xe, const RowArgs<N>& r) {
    using C = typename N::C;
    const RowPtr<N> p = row_ptr<N>(a, end, r.src, r.uh, r.ring, r.slot_stride, r.P, r.Pc, ax.N);
    unsigned mx = 0;
    each_mode<N, Ln>(ax, sm, end, xe, [&](int m, C F, C* at) {
        const double2 W = update_mode<N, WIDE>(a, g, sm.c, end, begin, m, F, p);
        if (begin) {
            *at = to_c(W, C());
            if constexpr (N::FX) mx = max(mx, fx_hi(*at));
        }
    });
    return mx;
}
// Row k0 of instance b along the last axis (1D: the only row).
template <class N> __device__ __forceinline__ RowArgs<N> row_args(const FsArgs& a, int b, int k0) {
    const int d = a.d, Nl = a.ax[d - 1].N;
    const size_t nrows = d == 1 ? 1 : (d == 2 ? (size_t)a.ax[0].N : (size_t)a.ax[0].N * a.ax[1].N);
    const size_t NPm = nrows * Nl, at = (size_t)b * NPm + (size_t)k0 * Nl, ph = (size_t)b * a.n_int * Nl;
    RowArgs<N> r;
    r.uh = a.uhat + at;
    r.src = a.uhat_src ? a.uhat_src + at : r.uh;
    r.ring = reinterpret_cast<typename N::C*>(a.ring) + (size_t)b * a.ring_slots * NPm + (size_t)k0 * Nl;
    r.slot_stride = NPm;
    r.P = a.ax[d - 1].P + ph;
    r.Pc = PhaseTab<N>::get(a.ax[d - 1]) + ph;
    return r;
}
// (Few arguments: what the call keeps alive counts against the registers of the
// fixed-point form.)
template <class N, class Ln>
__device__ __noinline__ unsigned update_modes_wide(const FsArgs& a, int flags, int xe) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int b = a.d == 1 ? blockIdx.x : blockIdx.y, k0 = a.d == 1 ? 0 : blockIdx.x;
    return update_modes<N, Ln, true>(a, a.ax[a.d - 1], *reinterpret_cast<typename Ln::Sm*>(sm_raw), FS_WIDE, flags & FS_ROW_END,
                                     flags & FS_ROW_BEGIN, xe, row_args<N>(a, b, k0));
}

// Row factor a_i of interval a.interval[i] of row k0 (1D: 1): P0 (2D), P0 P1 of axes 0 and 1 (3D).
template <bool WIDE> __device__ __forceinline__ int4 row_phase(const FsArgs& a, int g, int b, int k0, int i) {
    if (a.d == 1) return phase_one<WIDE>(g);
    const int iv = a.interval[i], N0 = a.ax[0].N;
    const int4* P0 = a.ax[0].P + (size_t)b * a.n_int * N0;
    if (a.d == 2) return __ldg(&P0[(size_t)iv * N0 + k0]);
    const int NA = a.ax[1].N, i0 = k0 / NA, i1 = k0 - i0 * NA;
    const int4* PA = a.ax[1].P + (size_t)b * a.n_int * NA;
    return phase_mul<WIDE>(__ldg(&P0[(size_t)iv * N0 + i0]), __ldg(&PA[(size_t)iv * NA + i1]), g);
}
template <class N, class Ln>
__device__ __noinline__ void row_factors_wide(const FsArgs& a) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int b = a.d == 1 ? blockIdx.x : blockIdx.y, k0 = a.d == 1 ? 0 : blockIdx.x;
    row_factors<N, true>(a, FS_WIDE, *reinterpret_cast<typename Ln::Sm*>(sm_raw), Ln::G::T,
                         [&](int i) { return row_phase<true>(a, FS_WIDE, b, k0, i); });
}

template <class N, int M, int R>
__global__ void __launch_bounds__((Geo<M, R>::T), (min_blocks<N, Geo<M, R>>())) k_fs_1d(const __grid_constant__ FsArgs a, int mode) {
    using Ln = Line<N, M, R>;
    using G = typename Ln::G;
    using C = typename N::C;
    using Rl = typename cx_traits<C>::real;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    typename Ln::Sm& sm = *reinterpret_cast<typename Ln::Sm*>(sm_raw);
    const FsAxis& ax = a.ax[0];
    const int b = blockIdx.x, Nm = ax.N, g = __ldg(&a.g[b]);
    const double vf = a.tfac[(size_t)b * a.ntf + a.tf];
    const double* V0 = a.V0 + (size_t)b * a.vstride;
    C f[G::FPT];
    int xe;
    if (mode == FS_1D_FWD_ONLY) {
#pragma unroll
        for (int p = 0; p < G::FPT; ++p) {
            const int j = threadIdx.x + p * G::T;
            f[p] = czero<C>();
            if (j < M) {
                const double2 u = a.usrc[(size_t)b * M + j];
                f[p] = cvt<C>(a.mulV ? cscale(u, vf * V0[j]) : u);
            }
        }
        const auto E = Ln::put_grid(f, sm, ax);
        Ln::forward(sm, ax, E, xe);
        each_mode<N, Ln>(ax, sm, true, xe, [&](int m, C F, C*) { store_fwd(a, (size_t)b * a.fdst_bstride + m, F); });
        return;
    }
    if (g < FS_WIDE) row_factors<N, false>(a, g, sm, G::T, [&](int) { return phase_one<false>(g); });
    else row_factors_wide<N, Ln>(a);
    __syncthreads();
    const RowArgs<N> rp = row_args<N>(a, b, 0);
    const unsigned mx = g < FS_WIDE ? update_modes<N, Ln, false>(a, ax, sm, g, false, true, 0, rp)
                                    : update_modes_wide<N, Ln>(a, FS_ROW_BEGIN, 0);
    C y[G::FPT];
    Ln::inverse(sm, mx, y, ax);
    const double hm0 = a.h * a.mu[0];
#pragma unroll
    for (int p = 0; p < G::FPT; ++p) {
        const int j = threadIdx.x + p * G::T;
        f[p] = czero<C>();
        if (j < M) {
            const double V = vf * V0[j];
            const C u = implicit_solve(y[p], (Rl)(hm0 * V));
            a.u[(size_t)b * M + j] = cvt<double2>(u);
            f[p] = cscale(u, (Rl)V);
        }
    }
    __syncthreads();                 // every thread has read its y
    const auto E = Ln::put_grid(f, sm, ax);
    Ln::forward(sm, ax, E, xe);
    update_modes<N, Ln, false>(a, ax, sm, g, true, false, xe, rp);      // (no phases)
}

template <class N, int M, int R>
__global__ void __launch_bounds__((Geo<M, R>::T), (min_blocks<N, Geo<M, R>>())) k_fs_row(const __grid_constant__ FsArgs a, int flags) {
    using Ln = Line<N, M, R>;
    using G = typename Ln::G;
    using C = typename N::C;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    typename Ln::Sm& sm = *reinterpret_cast<typename Ln::Sm*>(sm_raw);
    const bool d3 = a.d == 3;
    const FsAxis& ax = a.ax[d3 ? 2 : 1];                // the line axis (the last one)
    const int k0 = blockIdx.x, b = blockIdx.y;           // k0: the row (k0 N1 + k1 in 3D)
    const int N0 = a.ax[0].N, N1 = ax.N, g = __ldg(&a.g[b]);
    const int nrows = d3 ? N0 * a.ax[1].N : N0;
    const RowArgs<N> rp = row_args<N>(a, b, k0);
    C* zrow = reinterpret_cast<C*>(a.Z) + ((size_t)b * nrows + k0) * M;
    const bool end = flags & FS_ROW_END, begin = flags & FS_ROW_BEGIN;
    if (begin) {
        if (g < FS_WIDE) row_factors<N, false>(a, g, sm, G::T, [&](int i) { return row_phase<false>(a, g, b, k0, i); });
        else row_factors_wide<N, Ln>(a);
    }
    // the row's state and history on their way to the L2 while the transform runs
    if (begin) {
        for (int off = (int)threadIdx.x * 128; off < N1 * 16; off += G::T * 128) {
            asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char*>(rp.src) + off));
            if (off < N1 * (int)sizeof(C))
                for (int j = 0; j < a.nhist; ++j)
                    if (!(end && a.hist_slot[j] == a.out_slot))
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(
                            reinterpret_cast<const char*>(rp.ring + (size_t)a.hist_slot[j] * rp.slot_stride) + off));
        }
    }
    int xe = 0;
    if (end || (flags & FS_ROW_FWD_ONLY)) {
        C f[G::FPT];
#pragma unroll
        for (int p = 0; p < G::FPT; ++p) {
            const int j = threadIdx.x + p * G::T;
            f[p] = j < M ? zrow[j] : czero<C>();
        }
        const auto E = Ln::put_grid(f, sm, ax);
        Ln::forward(sm, ax, E, xe);
        if (flags & FS_ROW_FWD_ONLY) {
            const size_t base = (size_t)b * a.fdst_bstride + (size_t)k0 * N1;
            each_mode<N, Ln>(ax, sm, true, xe, [&](int m, C F, C*) { store_fwd(a, base + m, F); });
            return;
        }
    } else {
        __syncthreads();             // sm.c
    }
    const unsigned mx = g < FS_WIDE ? update_modes<N, Ln, false>(a, ax, sm, g, end, begin, xe, rp)
                                    : update_modes_wide<N, Ln>(a, flags, xe);
    if (!begin) return;
    C y[G::FPT];
    Ln::inverse(sm, mx, y, ax);
#pragma unroll
    for (int p = 0; p < G::FPT; ++p) {
        const int j = threadIdx.x + p * G::T;
        if (j < M) zrow[j] = y[p];
    }
}

// This thread's modes of a line z (stride n elements) as inputs of the inverse
// transform (all loads in flight together).
template <class N, class Ln>
__device__ __forceinline__ unsigned load_modes(const typename N::C* z, size_t n, typename Ln::Sm& sm, const FsAxis& ax) {
    using C = typename N::C;
    C x[Ln::NV];
#pragma unroll
    for (int k = 0; k < Ln::NV; ++k) {
        const int m = Ln::mode(k, ax);
        x[k] = m >= 0 ? z[(size_t)m * n] : czero<C>();
    }
    for (int d = threadIdx.x; d < ax.ND; d += Ln::G::T) sm.d[d] = z[(size_t)(ax.NE + d) * n];
    unsigned mx = 0;
#pragma unroll
    for (int k = 0; k < Ln::NV; ++k) {
        if (Ln::mode(k, ax) >= 0) *reinterpret_cast<C*>(Ln::slot(sm, k)) = x[k];
        if constexpr (N::FX) mx = max(mx, fx_hi(x[k]));
    }
    return mx;
}

template <class N, int M, int R>
__global__ void __launch_bounds__((Geo<M, R>::T), (min_blocks<N, Geo<M, R>>())) k_fs_phys(const __grid_constant__ FsArgs a, int from_usrc) {
    using Ln = Line<N, M, R>;
    using G = typename Ln::G;
    using C = typename N::C;
    using Rl = typename cx_traits<C>::real;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    typename Ln::Sm& sm = *reinterpret_cast<typename Ln::Sm*>(sm_raw);
    const FsAxis& ax = a.ax[0];
    const int j1 = blockIdx.x, b = blockIdx.y;          // j1: the column (j1 M2 + j2 in 3D)
    const bool d3 = a.d == 3;
    const int M1 = d3 ? a.ax[1].M * a.ax[2].M : a.ax[1].M, N0 = ax.N;
    C* zcol = reinterpret_cast<C*>(d3 ? a.Y : a.Z) + (size_t)b * N0 * M1 + j1;
    const size_t NX = (size_t)M * M1;
    const double vf = a.tfac[(size_t)b * a.ntf + a.tf];
    const double* V0 = a.V0 + (size_t)b * a.vstride;
    C f[G::FPT];
    if (!from_usrc) {
        C y[G::FPT];
        const unsigned mx = load_modes<N, Ln>(zcol, (size_t)M1, sm, ax);
        Ln::inverse(sm, mx, y, ax);
        const double hm0 = a.h * a.mu[0];
#pragma unroll
        for (int p = 0; p < G::FPT; ++p) {
            const int j0 = threadIdx.x + p * G::T;
            f[p] = czero<C>();
            if (j0 < M) {
                const size_t g = (size_t)j0 * M1 + j1;
                const double V = vf * V0[g];
                const C u = implicit_solve(y[p], (Rl)(hm0 * V));
                a.u[(size_t)b * NX + g] = cvt<double2>(u);
                f[p] = cscale(u, (Rl)V);
            }
        }
        __syncthreads();             // every thread has read its y
    } else {
#pragma unroll
        for (int p = 0; p < G::FPT; ++p) {
            const int j0 = threadIdx.x + p * G::T;
            f[p] = czero<C>();
            if (j0 < M) {
                const size_t g = (size_t)j0 * M1 + j1;
                const double2 u = a.usrc[(size_t)b * NX + g];
                f[p] = cvt<C>(a.mulV ? cscale(u, vf * V0[g]) : u);
            }
        }
    }
    int xe;
    const auto E = Ln::put_grid(f, sm, ax);
    Ln::forward(sm, ax, E, xe);
    each_mode<N, Ln>(ax, sm, true, xe, [&](int m, C F, C*) { zcol[(size_t)m * M1] = F; });
}

// 3D, axis 1: line (k0, j2) between the N1 modes Z[b][k0][.][j2] and the M1
// grid values Y[b][k0][.][j2] (both with stride M2).
template <class N, int M, int R>
__global__ void __launch_bounds__((Geo<M, R>::T), (min_blocks<N, Geo<M, R>>())) k_fs_mid(const __grid_constant__ FsArgs a, int dir) {
    using Ln = Line<N, M, R>;
    using G = typename Ln::G;
    using C = typename N::C;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    typename Ln::Sm& sm = *reinterpret_cast<typename Ln::Sm*>(sm_raw);
    const FsAxis& ax = a.ax[1];
    const int j2 = blockIdx.x, k0 = blockIdx.y, b = blockIdx.z;
    const int M2 = a.ax[2].M, N0 = a.ax[0].N, N1 = ax.N;
    C* zl = reinterpret_cast<C*>(a.Z) + ((size_t)b * N0 + k0) * N1 * M2 + j2;
    C* yl = reinterpret_cast<C*>(a.Y) + ((size_t)b * N0 + k0) * M * M2 + j2;
    C f[G::FPT];
    if (dir == FS_MID_INV) {
        const unsigned mx = load_modes<N, Ln>(zl, (size_t)M2, sm, ax);
        Ln::inverse(sm, mx, f, ax);
#pragma unroll
        for (int p = 0; p < G::FPT; ++p) {
            const int j = threadIdx.x + p * G::T;
            if (j < M) yl[(size_t)j * M2] = f[p];
        }
    } else {
#pragma unroll
        for (int p = 0; p < G::FPT; ++p) {
            const int j = threadIdx.x + p * G::T;
            f[p] = j < M ? yl[(size_t)j * M2] : czero<C>();
        }
        int xe;
        const auto E = Ln::put_grid(f, sm, ax);
        Ln::forward(sm, ax, E, xe);
        each_mode<N, Ln>(ax, sm, true, xe, [&](int m, C F, C*) { zl[(size_t)m * M2] = F; });
    }
}

// Dynamic shared memory of the kernel and the largest shared-memory carve-out
// (several CTAs per SM).
template <class K>
cudaError_t prepare(K kernel, size_t sm) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    return e;
}

template <class N, int M, int R>
cudaError_t launch_mr(const FsArgs& a, int which, int flag, cudaStream_t s) {
    using G = Geo<M, R>;
    constexpr size_t sm = sizeof(Smem<N, G>);
    static DeviceOnce once[4];
    cudaError_t e = cudaSuccess;
    auto ready = [&](auto kernel) {
        e = once[which]([&] { return prepare(kernel, sm); });
        return e == cudaSuccess;
    };
    if (which == 0) {
        if (!ready(k_fs_1d<N, M, R>)) return e;
        k_fs_1d<N, M, R><<<a.B, G::T, sm, s>>>(a, flag);
    } else if (which == 1) {
        if (!ready(k_fs_row<N, M, R>)) return e;
        const unsigned rows = a.d == 3 ? (unsigned)(a.ax[0].N * a.ax[1].N) : (unsigned)a.ax[0].N;
        k_fs_row<N, M, R><<<dim3(rows, a.B), G::T, sm, s>>>(a, flag);
    } else if (which == 2) {
        if (!ready(k_fs_phys<N, M, R>)) return e;
        const unsigned cols = a.d == 3 ? (unsigned)(a.ax[1].M * a.ax[2].M) : (unsigned)a.ax[1].M;
        k_fs_phys<N, M, R><<<dim3(cols, a.B), G::T, sm, s>>>(a, flag);
    } else {
        if (!ready(k_fs_mid<N, M, R>)) return e;
        k_fs_mid<N, M, R><<<dim3(a.ax[2].M, a.ax[0].N, a.B), G::T, sm, s>>>(a, flag);
    }
    return cudaGetLastError();
}

// (M, R) pairs built: M = 32..512, R = 4, 8, 16, nu = M R <= 4096.
template <class N>
cudaError_t dispatch(const FsArgs& a, const FsAxis& ax, int which, int flag, cudaStream_t s) {
#define FS_FOR_R(M_)                                                                               \
    if (R == 4) return launch_mr<N, M_, 4>(a, which, flag, s);                                   \
    if (R == 8) return launch_mr<N, M_, 8>(a, which, flag, s);                                   \
    if (R == 16 && M_ * 16 <= 4096) return launch_mr<N, M_, (M_ * 16 <= 4096 ? 16 : 8)>(a, which, flag, s);
    const int M = ax.M, R = ax.R;
    switch (M) {
        case 32: { FS_FOR_R(32) break; }
        case 64: { FS_FOR_R(64) break; }
        case 128: { FS_FOR_R(128) break; }
        case 256: { FS_FOR_R(256) break; }
        case 512: { FS_FOR_R(512) break; }
        default: break;
    }
#undef FS_FOR_R
    return cudaErrorInvalidValue;
}

// which: 0 = 1D step, 1 = row pass (last axis), 2 = phys pass (axis 0), 3 = axis-1 pass (3D)
inline const FsAxis& axis_of(const FsArgs& a, int which) {
    return which == 1 ? a.ax[a.d - 1] : (which == 3 ? a.ax[1] : a.ax[0]);
}

}  // namespace fs
}  // namespace tdse
