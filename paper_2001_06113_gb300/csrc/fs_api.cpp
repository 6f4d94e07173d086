// Free-space orchestration (bc = TDSE_FREE): the contour rule of Sec. 3.4 and
// 4.1, the transform and phase tables, the workspace layout and the launch
// sequence of the start-up (Richardson on u^ and u, Remark highorderfs) and
// of the Adams steps.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "alpert_rules.h"
#include "ctx.h"
#include "fsargs.h"
#include "fx.cuh"
#include "kargs.h"

using namespace tdse;

namespace {

constexpr long double kPiL = 3.141592653589793238462643383279502884L;

const AlpertRule* find_alpert(int p) {
    for (const AlpertRule& r : kAlpertRules)
        if (r.p == p) return &r;
    return nullptr;
}

// e^{i theta} with theta reduced to [-pi, pi] in long double first, so that
// large phases (|theta| up to ~ K) lose no accuracy.
void cis(long double theta, double& c, double& s) {
    long double r = fmodl(theta, 2.0L * kPiL);
    if (r > kPiL) r -= 2.0L * kPiL;
    if (r < -kPiL) r += 2.0L * kPiL;
    c = std::cos((double)r);
    s = std::sin((double)r);
}

// Nodes and weights of one axis (Sec. 3.4): E1, A1, C, A3, E3.
bool build_rule(FsAxisHost& A, int M, int nu, int p, int q, int n_r, double H) {
    const AlpertRule* ar = find_alpert(p);
    if (!ar) return false;
    A.M = M;
    A.nu = nu;
    A.R = nu / M;
    A.p = p;
    A.kappa = ar->kappa;
    A.q = q;
    A.n_r = n_r;
    A.H = H;
    A.NE = nu / 2 - 2 * A.kappa + 1;                 // nu = 2 (NE + 2 kappa - 1)
    if (A.NE <= M / 2) return false;                 // the blocks must reach beyond |Re zeta| = pi M / 2 - ...
    A.K = H + M_PI * M / 2.0;
    A.h = (A.K - H) / (A.NE + 2 * A.kappa - 1);
    A.NC = q * (n_r == 0 ? 1 : 2 * n_r);
    A.ND = 2 * p + A.NC;
    A.N = 2 * A.NE + A.ND;
    if (A.ND > FS_MAX_ND) return false;
    A.zeta.clear();
    A.w.clear();
    auto push = [&](double zr, double zi, double wr, double wi) {
        A.zeta.push_back(zr);
        A.zeta.push_back(zi);
        A.w.push_back(wr);
        A.w.push_back(wi);
    };
    const double h = A.h;
    // E1: reflection of E3 (zeta -> -zeta), ascending real part
    for (int i = 0; i < A.NE; ++i) push(-((H + A.kappa * h) + (A.NE - 1 - i) * h), H, h, 0.0);
    // A1: reflection of the Alpert nodes on Gamma_3
    for (int k = p - 1; k >= 0; --k) push(-(H + ar->x[k] * h), H, h * ar->w[k], 0.0);
    // C: composite q-point Gauss-Legendre on Gamma_2, zeta = (1 - i) tau, d zeta = (1 - i) d tau,
    // panels [-H, H] (n_r = 0) or dyadic toward 0: edges +-H / 2^(n_r - k), k = 1..n_r, and 0
    std::vector<double> gx, gw;
    gauss_legendre(q, gx, gw);
    std::vector<int> order(q);
    for (int i = 0; i < q; ++i) order[i] = i;
    std::sort(order.begin(), order.end(), [&](int a, int b) { return gx[a] < gx[b]; });
    std::vector<double> edges;
    if (n_r == 0) {
        edges = {-H, H};
    } else {
        std::vector<double> pos = {0.0};
        for (int k = 1; k <= n_r; ++k) pos.push_back(H / std::ldexp(1.0, n_r - k));
        for (int k = (int)pos.size() - 1; k >= 1; --k) edges.push_back(-pos[k]);
        for (double v : pos) edges.push_back(v);
    }
    for (size_t e = 0; e + 1 < edges.size(); ++e) {
        const double a = edges[e], b = edges[e + 1];
        for (int i : order) {
            const double tau = 0.5 * (b - a) * gx[i] + 0.5 * (a + b);
            const double wt = 0.5 * (b - a) * gw[i];
            push(tau, -tau, wt, -wt);
        }
    }
    // A3 and E3 on Gamma_3: tau - iH
    for (int k = 0; k < p; ++k) push(H + ar->x[k] * h, -H, h * ar->w[k], 0.0);
    for (int i = 0; i < A.NE; ++i) push((H + A.kappa * h) + i * h, -H, h, 0.0);
    return (int)A.zeta.size() == 2 * A.N;
}

struct AxisTables {
    std::vector<double> zeta, preI, postI, preF, postF, Gd, Fd, tw;
    std::vector<double> Lf, Li, Tc, TcW;   // Chebyshev form of the C-type transforms (NT > 0)
};

// Chebyshev form of the C-type transforms (Sec. 4.1).  For a grid point x the
// function tau -> e^{s (1+i) tau x} (s = -1 forward: e^{-i zeta x}; s = +1
// inverse: e^{+i zeta x}, zeta = (1 - i) tau) on [-H, H] is replaced by its
// NT-point Chebyshev interpolant sum_l c_l T_l(tau / H), the coefficients from
// the values at the Chebyshev points tau_m = H cos(pi (m + 1/2) / NT):
//   c_l = (2 / NT) sum_m g(tau_m) cos(l pi (m + 1/2) / NT),  c_0 halved.
// Long double throughout, rounded once.
struct ChebPoints {
    int NT;
    std::vector<long double> u, cosl_;   // cos(th_m), cos(l th_m) [m][l]
    ChebPoints(int nt) : NT(nt), u(nt), cosl_((size_t)nt * nt) {
        for (int m = 0; m < nt; ++m) {
            const long double th = kPiL * (m + 0.5L) / nt;
            u[m] = cosl(th);
            for (int l = 0; l < nt; ++l) cosl_[(size_t)m * nt + l] = cosl(l * th);
        }
    }
};
void cheb_coeffs(long double x, int s, long double H, const ChebPoints& P, std::vector<long double>& cr,
                 std::vector<long double>& ci) {
    const int NT = P.NT;
    cr.assign(NT, 0.0L);
    ci.assign(NT, 0.0L);
    for (int m = 0; m < NT; ++m) {
        const long double tau = H * P.u[m];
        const long double mag = expl(s * tau * x), ang = s * tau * x;   // e^{s tau x} e^{i s tau x}
        const long double gr = mag * cosl(ang), gi = mag * sinl(ang);
        const long double* cl = &P.cosl_[(size_t)m * NT];
        for (int l = 0; l < NT; ++l) {
            cr[l] += gr * cl[l];
            ci[l] += gi * cl[l];
        }
    }
    for (int l = 0; l < NT; ++l) {
        cr[l] *= 2.0L / NT;
        ci[l] *= 2.0L / NT;
    }
    cr[0] *= 0.5L;
    ci[0] *= 0.5L;
}

// T_l(u), l = 0..NT-1, by the three-term recurrence
void cheb_T(long double u, int NT, std::vector<long double>& T) {
    T.assign(NT, 0.0L);
    T[0] = 1.0L;
    if (NT > 1) T[1] = u;
    for (int l = 2; l < NT; ++l) T[l] = 2.0L * u * T[l - 1] - T[l - 2];
}

// Smallest NT (8..FS_MAX_NT, even) whose interpolants reproduce e^{-+i zeta x}
// at every C node to 4 units of FP64 rounding of the largest value, checked
// at every 16th grid point and at both ends of the grid (the interpolation
// error of e^{a tau} grows with |a| = sqrt(2) |x|, largest at the ends); 0 if
// none does.
int choose_nt(const FsAxisHost& A) {
    const int p = A.p, NC = A.NC, M = A.M, NE = A.NE;
    const long double H = A.H;
    std::vector<long double> cr, ci, T;
    for (int NT = 8; NT <= FS_MAX_NT; NT += 2) {
        const ChebPoints P(NT);
        long double err = 0.0L, big = 0.0L;
        for (int j = 0; j < M; j = (j + 16 < M || j == M - 1) ? j + 16 : M - 1) {
            const long double x = -1.0L + 2.0L * j / M;
            for (int sg = -1; sg <= 1; sg += 2) {
                cheb_coeffs(x, sg, H, P, cr, ci);
                for (int k = 0; k < NC; ++k) {
                    const long double tau = A.zeta[2 * (NE + p + k)];
                    cheb_T(tau / H, NT, T);
                    long double vr = 0.0L, vi = 0.0L;
                    for (int l = 0; l < NT; ++l) {
                        vr += cr[l] * T[l];
                        vi += ci[l] * T[l];
                    }
                    const long double mag = expl(sg * tau * x), ang = sg * tau * x;
                    const long double gr = mag * cosl(ang), gi = mag * sinl(ang);
                    err = fmaxl(err, hypotl(vr - gr, vi - gi));
                    big = fmaxl(big, mag);
                }
            }
        }
        if (err <= 4.0L * 2.220446049250313e-16L * big) return NT;
    }
    return 0;
}

void make_cheb_tables(const FsAxisHost& A, AxisTables& T) {
    const int M = A.M, NT = A.NT, NC = A.NC, NE = A.NE, p = A.p;
    const long double H = A.H;
    std::vector<long double> cr, ci, Tl;
    const ChebPoints P(NT);
    T.Lf.assign((size_t)2 * NT * M, 0.0);
    T.Li.assign((size_t)2 * NT * M, 0.0);
    for (int j = 0; j < M; ++j) {
        const long double x = -1.0L + 2.0L * j / M;
        cheb_coeffs(x, -1, H, P, cr, ci);
        for (int l = 0; l < NT; ++l) {
            T.Lf[2 * ((size_t)l * M + j)] = (double)(cr[l] * 2.0L / M);
            T.Lf[2 * ((size_t)l * M + j) + 1] = (double)(ci[l] * 2.0L / M);
        }
        cheb_coeffs(x, +1, H, P, cr, ci);
        for (int l = 0; l < NT; ++l) {
            T.Li[2 * ((size_t)l * M + j)] = (double)cr[l];
            T.Li[2 * ((size_t)l * M + j) + 1] = (double)ci[l];
        }
    }
    T.Tc.assign((size_t)NC * NT, 0.0);
    T.TcW.assign((size_t)2 * NT * NC, 0.0);
    const long double inv2pi = 1.0L / (2.0L * kPiL);
    for (int k = 0; k < NC; ++k) {
        const int m = NE + p + k;
        cheb_T((long double)A.zeta[2 * m] / H, NT, Tl);
        const long double wr = A.w[2 * m] * inv2pi, wi = A.w[2 * m + 1] * inv2pi;
        for (int l = 0; l < NT; ++l) {
            T.Tc[(size_t)k * NT + l] = (double)Tl[l];
            T.TcW[2 * ((size_t)l * NC + k)] = (double)(Tl[l] * wr);
            T.TcW[2 * ((size_t)l * NC + k) + 1] = (double)(Tl[l] * wi);
        }
    }
}

// Host tables of one axis (fsargs.h FsAxis), in FP64 from long double phases.
AxisTables make_tables(const FsAxisHost& A) {
    AxisTables T;
    const int M = A.M, R = A.M > 256 ? 2 * A.R : A.R, nu = A.nu, NE = A.NE, ND = A.ND;   // R lines per block (freespace.cuh)
    const long double h = A.h;
    T.zeta = A.zeta;
    auto put = [](std::vector<double>& v, double mag, long double theta) {
        double c, s;
        cis(theta, c, s);
        v.push_back(mag * c);
        v.push_back(mag * s);
    };
    const long double inv2pi = 1.0L / (2.0L * kPiL);
    // block origins zeta0 (E1: first node; E3: node NE + ND)
    const double z0r[2] = {A.zeta[0], A.zeta[2 * (NE + ND)]};
    const double z0i[2] = {A.zeta[1], A.zeta[2 * (NE + ND) + 1]};
    for (int b = 0; b < 2; ++b)
        for (int i = 0; i < NE; ++i) put(T.preI, (double)(h * inv2pi), -(long double)i * h);
    for (int b = 0; b < 2; ++b)
        for (int j = 0; j < M; ++j) {
            const double x = -1.0 + 2.0 * j / M;
            for (int s = 0; s < R; ++s) {
                const long double tw = 2.0L * kPiL * (long double)(((long long)j * s) % nu) / nu;
                // e^{i zeta0 x} = e^{-Im(zeta0) x} e^{i Re(zeta0) x}
                put(T.postI, std::exp(-z0i[b] * x), (long double)z0r[b] * x + tw);
                put(T.preF, (2.0 / M) * std::exp(z0i[b] * x), -(long double)z0r[b] * x - tw);
            }
        }
    for (int b = 0; b < 2; ++b)
        for (int i = 0; i < NE; ++i) put(T.postF, 1.0, (long double)i * h);
    for (int dd = 0; dd < ND; ++dd) {
        const int m = NE + dd;
        const double zr = A.zeta[2 * m], zi = A.zeta[2 * m + 1];
        const double wr = A.w[2 * m] / (2.0 * M_PI), wi = A.w[2 * m + 1] / (2.0 * M_PI);
        for (int j = 0; j < M; ++j) {
            const double x = -1.0 + 2.0 * j / M;
            double c, s;
            cis((long double)zr * x, c, s);
            const double e = std::exp(-zi * x);
            // (w / 2pi) e^{i zeta x}
            const double gr = e * c, gi = e * s;
            T.Gd.push_back(wr * gr - wi * gi);
            T.Gd.push_back(wr * gi + wi * gr);
            // (2/M) e^{-i zeta x} = (2/M) e^{zi x} (c - i s)
            const double f = (2.0 / M) / e;
            T.Fd.push_back(f * c);
            T.Fd.push_back(-f * s);
        }
    }
    const int MF = A.M > 256 ? M / 2 : M;        // transform length
    for (int m = 0; m < MF; ++m) put(T.tw, 1.0, -2.0L * kPiL * m / MF);
    if (A.NT > 0) make_cheb_tables(A, T);
    return T;
}

FsArgs fs_base(const tdse_ctx* c) {
    const FsState& F = c->F;
    FsArgs a{};
    a.B = c->B;
    a.d = c->d;
    for (int x = 0; x < 3; ++x) {
        FsAxis& X = a.ax[x];
        if (x >= c->d) {
            X.M = 1;
            X.N = 1;
            continue;
        }
        const FsAxisHost& A = F.ax[x];
        X.M = A.M;
        X.R = A.R;
        X.nu = A.nu;
        X.NE = A.NE;
        X.ND = A.ND;
        X.N = A.N;
        X.preI = c->P<int4>(F.off.preI[x]);
        X.postI = c->P<int4>(F.off.postI[x]);
        X.preF = c->P<int4>(F.off.preF[x]);
        X.postF = c->P<int4>(F.off.postF[x]);
        X.Gd = c->P<int4>(F.off.Gd[x]);
        X.Fd = c->P<int4>(F.off.Fd[x]);
        X.tw = c->P<int4>(F.off.tw[x]);
        X.P = c->P<int4>(F.off.P[x]);
        X.xI = A.xI;
        X.xj = c->P<int>(F.off.xj[x]);
        X.p = A.p;
        X.NC = A.NC;
        X.NT = A.NT;
        if (A.NT > 0) {
            X.Lf = c->P<int4>(F.off.Lf[x]);
            X.Li = c->P<int4>(F.off.Li[x]);
            X.Tc = c->P<double>(F.off.Tc[x]);
            X.TcW = c->P<double2>(F.off.TcW[x]);
            if (F.f32) {
                X.Lf_f = c->P<float2>(F.off.Lf_f[x]);
                X.Li_f = c->P<float2>(F.off.Li_f[x]);
                X.Tc_f = c->P<float>(F.off.Tc_f[x]);
                X.TcW_f = c->P<float2>(F.off.TcW_f[x]);
            }
        }
        if (F.f32) {
            X.preI_f = c->P<float2>(F.off.preI_f[x]);
            X.postI_f = c->P<float2>(F.off.postI_f[x]);
            X.preF_f = c->P<float2>(F.off.preF_f[x]);
            X.postF_f = c->P<float2>(F.off.postF_f[x]);
            X.Gd_f = c->P<float2>(F.off.Gd_f[x]);
            X.Fd_f = c->P<float2>(F.off.Fd_f[x]);
            X.tw_f = c->P<float2>(F.off.tw_f[x]);
            X.P_f = c->P<float2>(F.off.P_f[x]);
        }
    }
    a.g = c->P<int>(F.off.g);
    a.n_int = c->n_int;
    a.uhat = c->P<double2>(F.off.uhat);
    a.ring = c->P<double2>(F.off.ring);
    a.ring_slots = c->RS;
    a.Z = F.off.Z ? c->P<double2>(F.off.Z) : nullptr;
    a.Y = F.off.Y ? c->P<double2>(F.off.Y) : nullptr;
    a.u = c->P<double2>(F.off.u);
    a.V0 = c->P<double>(F.off.V0);
    a.vstride = c->vshared ? 0 : (size_t)c->vrows * F.NX;
    a.tfac = c->P<double>(F.off.tfac);
    a.ntf = c->ntf;
    return a;
}

// The launch evaluates V at t = tf dt / 8 (with a potential table: that row).
void set_time(const tdse_ctx* c, FsArgs& a, int tf) {
    a.tf = tf;
    a.V0 = c->P<double>(c->F.off.V0) + vrow(c, tf) * c->F.NX;
}

// Step size and weights of a step with n history terms.
void set_weights(FsArgs& a, double h, const double* mu, int n) {
    auto factor = [](double x, int2& w) { fx_limbs(std::llround(std::ldexp(x, 61)), w.x, w.y); };
    a.nhist = n;
    a.h = h;
    const double f[2] = {1.0, FX_WIDEN};
    for (int i = 0; i < 2; ++i) {
        a.up_h[i] = h * f[i];
        a.up_hmu0[i] = h * mu[0] * f[i];
    }
    for (int j = 0; j <= n; ++j) {
        a.mu[j] = mu[j];
        factor(0.5 * mu[j], a.mu_w[j]);
    }
}

// Ring slot `slot` of a ring with rsz-byte elements (as the kernels' double2* field).
double2* ring_at(const tdse_ctx* c, size_t ring_off, size_t elems) {
    return reinterpret_cast<double2*>(c->P<char>(ring_off) + elems * c->rsz);
}

// Grid values usrc (times V(t_tf) if mulV) -> mode space: into the FP64 state
// (to_ring = 0) or a ring slot in the ring's element type (to_ring = 1), instance
// b at fdst + b bstride elements.
tdse_status forward_to(tdse_ctx* c, const double2* usrc, int mulV, int tf, double2* fdst, size_t bstride,
                       int to_ring, cudaStream_t s) {
    FsArgs a = fs_base(c);
    a.usrc = usrc;
    a.mulV = mulV;
    set_time(c, a, tf);
    a.fdst = fdst;
    a.fdst_bstride = bstride;
    a.fdst_ring = to_ring;
    const int f32 = c->F.f32 ? 1 : 0;
    if (c->d == 1) {
        TDSE_CK(c, launch_fs_1d(a, FS_1D_FWD_ONLY, f32, s));
    } else {
        TDSE_CK(c, launch_fs_phys(a, 1, f32, s));
        if (c->d == 3) TDSE_CK(c, launch_fs_mid(a, FS_MID_FWD, f32, s));
        TDSE_CK(c, launch_fs_row(a, FS_ROW_FWD_ONLY, f32, s));
    }
    return TDSE_OK;
}

// The part of a 2D / 3D step between the row passes: the grid work along
// axis 0 (3D: between the inverse and the forward transform along axis 1).
tdse_status grid_part(tdse_ctx* c, const FsArgs& a, int f32, cudaStream_t s) {
    if (c->d == 3) TDSE_CK(c, launch_fs_mid(a, FS_MID_INV, f32, s));
    TDSE_CK(c, launch_fs_phys(a, 0, f32, s));
    if (c->d == 3) TDSE_CK(c, launch_fs_mid(a, FS_MID_FWD, f32, s));
    return TDSE_OK;
}

tdse_status fs_init(tdse_ctx* c, cudaStream_t s) {
    const FsState& F = c->F;
    double2* u = c->P<double2>(F.off.u);
    tdse_status st = forward_to(c, u, 0, 0, c->P<double2>(F.off.uhat), F.NM, 0, s);
    if (st != TDSE_OK) return st;
    st = forward_to(c, u, 1, 0, ring_at(c, F.off.ring, (size_t)slot_of(c, 0) * F.NM), (size_t)c->RS * F.NM, 1, s);
    if (st != TDSE_OK) return st;
    c->inited = true;
    return TDSE_OK;
}

// Steps first..last of a chain, step i described by args(i), the begin of the
// first by begin().  2D / 3D: row
// begin, (grid part, row end + begin) x (last - first), grid part, row end;
// the end of step i runs with the arguments of i + 1 and the ring slot of i.
template <class Begin, class Args>
tdse_status fs_chain(tdse_ctx* c, Begin begin, Args args, int first, int last, cudaStream_t s) {
    const int f32 = c->F.f32 ? 1 : 0;
    if (c->d == 1) {
        for (int i = first; i <= last; ++i) TDSE_CK(c, launch_fs_1d(args(i), FS_1D_STEP, f32, s));
        return TDSE_OK;
    }
    TDSE_CK(c, launch_fs_row(begin(), FS_ROW_BEGIN, f32, s));
    for (int i = first; i <= last; ++i) {
        const FsArgs a = args(i);
        tdse_status st = grid_part(c, a, f32, s);
        if (st != TDSE_OK) return st;
        FsArgs f = i < last ? args(i + 1) : a;
        f.out_slot = a.out_slot;
        TDSE_CK(c, launch_fs_row(f, i < last ? FS_ROW_END | FS_ROW_BEGIN : FS_ROW_END, f32, s));
    }
    return TDSE_OK;
}

// Start-up step n: L trapezoid chains with 1, 2, 4, .. sub-steps, Richardson
// combination of u^ and u, then (Vu)^(t_n) = forward(V(t_n) u).
tdse_status fs_startup_step(tdse_ctx* c, int n, cudaStream_t s) {
    const FsState& F = c->F;
    const size_t BM = (size_t)c->B * F.NM, BX = (size_t)c->B * F.NX;
    double2* cu = c->P<double2>(F.off.chain_uhat);
    double2* cx = c->P<double2>(F.off.chain_u);
    for (int ch = 0; ch < c->L; ++ch) {
        double2* cr = ring_at(c, F.off.chain_ring, ch * BM);
        if (c->d == 1) {
            TDSE_CK(c, cudaMemcpyAsync(cu + ch * BM, c->P<double2>(F.off.uhat), BM * 16, cudaMemcpyDeviceToDevice, s));
            TDSE_CK(c, launch_copy_slot(cr, c->P<void>(F.off.ring), c->RS, slot_of(c, n - 1), c->B, F.NM, c->rsz, s));
        }
        const int len = SUB >> ch, last = (1 << ch) - 1;
        auto sub = [&](int i) {     // trapezoid sub-step i of the chain
            FsArgs a = fs_base(c);
            a.uhat = cu + ch * BM;
            a.ring = cr;
            a.ring_slots = 1;
            a.u = cx + ch * BX;
            const double half[2] = {0.5, 0.5};
            set_weights(a, c->cfg.dt / (double)(1 << ch), half, 1);
            a.hist_slot[0] = 0;
            a.out_slot = 0;
            a.interval[0] = startup_interval(c, n, ch, i);
            set_time(c, a, SUB * (n - 1) + (i + 1) * len);
            return a;
        };
        // 2D / 3D: the first begin reads the state and the last (Vu)^ where they are
        auto first = [&]() {
            FsArgs a = sub(0);
            a.uhat_src = c->P<double2>(F.off.uhat);
            a.ring = c->P<double2>(F.off.ring);
            a.ring_slots = c->RS;
            a.hist_slot[0] = slot_of(c, n - 1);
            a.out_slot = -1;
            return a;
        };
        tdse_status st = fs_chain(c, first, sub, 0, last, s);
        if (st != TDSE_OK) return st;
    }
    TDSE_CK(c, launch_combine(c->P<void>(F.off.uhat), cu, BM, c->L, c->rich, BM, false, s));
    TDSE_CK(c, launch_combine(c->P<void>(F.off.u), cx, BX, c->L, c->rich, BX, false, s));
    return forward_to(c, c->P<double2>(F.off.u), 1, SUB * n, ring_at(c, F.off.ring, (size_t)slot_of(c, n) * F.NM),
                      (size_t)c->RS * F.NM, 1, s);
}

FsArgs adams_args(const tdse_ctx* c, int n) {
    FsArgs a = fs_base(c);
    set_weights(a, c->cfg.dt, c->mu, c->m - 1);
    for (int j = 1; j <= a.nhist; ++j) a.hist_slot[j - 1] = slot_of(c, n - j);
    a.out_slot = slot_of(c, n);
    for (int i = 0; i < a.nhist; ++i) a.interval[i] = main_interval(c, n - i);
    set_time(c, a, SUB * n);
    return a;
}

tdse_status fs_adams(tdse_ctx* c, int n0, int k, cudaStream_t s) {
    auto args = [&](int n) { return adams_args(c, n); };
    return fs_chain(c, [&]() { return args(n0 + 1); }, args, n0 + 1, n0 + k, s);
}

// FP64 residual of the implicit step just completed (step c->step, FP32
// transforms): W = u^ + i mu_0 h R_n, then the step's implicit part
// re-evaluated in FP64 (the FP64 kernels with no history term and a one-step
// phase of 1): u64 = inverse(W) / (1 + i mu_0 h V), R64 = forward(V u64),
// Wc = W - i mu_0 h R64; rho = mu_0 h ||R64 - R_n|| / ||u^||; where rho > tol
// (or is not finite) the step's results are replaced by the FP64 ones.
tdse_status fs_residual_check(tdse_ctx* c, cudaStream_t s) {
    const FsState& F = c->F;
    const int n = c->step;
    const double hm0 = c->cfg.dt * c->mu[0];
    const size_t rstride = (size_t)c->RS * F.NM;
    float2* ring_n = reinterpret_cast<float2*>(ring_at(c, F.off.ring, (size_t)slot_of(c, n) * F.NM));
    double2* uhat = c->P<double2>(F.off.uhat);
    double2* W = c->P<double2>(F.off.res_W);
    double2* R64 = c->P<double2>(F.off.res_R);
    double2* u64 = c->P<double2>(F.off.res_u);
    TDSE_CK(c, launch_fs_res_prep(W, uhat, ring_n, rstride, F.NM, c->B, hm0, s));
    FsArgs a = fs_base(c);
    a.uhat = W;                 // W in, W - i mu_0 h R64 out
    a.ring = R64;               // one FP64 slot: R64
    a.ring_slots = 1;
    a.u = u64;
    a.Z = F.off.Z64 ? c->P<double2>(F.off.Z64) : nullptr;
    a.Y = F.off.Y64 ? c->P<double2>(F.off.Y64) : nullptr;
    set_weights(a, c->cfg.dt, c->mu, 0);
    a.out_slot = 0;
    a.interval[0] = F.zero_iv;
    set_time(c, a, SUB * n);
    if (c->d == 1) {
        TDSE_CK(c, launch_fs_1d(a, FS_1D_STEP, 0, s));
    } else {
        TDSE_CK(c, launch_fs_row(a, FS_ROW_BEGIN, 0, s));
        tdse_status st = grid_part(c, a, 0, s);
        if (st != TDSE_OK) return st;
        TDSE_CK(c, launch_fs_row(a, FS_ROW_END, 0, s));
    }
    double* sums = c->P<double>(c->off.res_sums);
    int* flags = c->P<int>(c->off.res_flags);
    TDSE_CK(c, launch_fs_res_norms(R64, ring_n, rstride, uhat, F.NM, c->B, sums, s));
    TDSE_CK(c, launch_fs_res_decide(sums, c->B, hm0, c->res_tol, c->P<double>(c->off.res_rho), flags,
                                    c->P<int>(c->off.res_ncorr), s));
    TDSE_CK(c, launch_fs_res_apply(flags, c->B, F.NM, F.NX, uhat, W, ring_n, rstride, R64, c->P<double2>(F.off.u),
                                   u64, s));
    ++c->res_checks;
    return TDSE_OK;
}

}  // namespace

tdse_status fs_create(tdse_ctx* c) {
    const tdse_config& g = c->cfg;
    FsState& F = c->F;
    const int p = g.alpert_p == 0 ? 8 : g.alpert_p;
    if (!find_alpert(p)) return c->fail(TDSE_EINVAL, "alpert_p must be 4 or 8");
    if (g.gauss_q < 1 || g.gauss_q > 32) return c->fail(TDSE_EINVAL, "gauss_q must be in 1..32");
    if (g.n_r < 0 || g.n_r > 4) return c->fail(TDSE_EINVAL, "n_r must be in 0..4");
    if (!(g.H > 0.0) || !std::isfinite(g.H)) return c->fail(TDSE_EINVAL, "H must be positive");
    if (g.c_transform < TDSE_CT_AUTO || g.c_transform > TDSE_CT_CHEBYSHEV)
        return c->fail(TDSE_EINVAL, "c_transform: TDSE_CT_AUTO, TDSE_CT_DIRECT or TDSE_CT_CHEBYSHEV");
    F.f32 = g.precision == TDSE_MIXED;
    F.NM = 1;
    F.NX = 1;
    for (int x = 0; x < c->d; ++x) {
        const int M = x < 2 ? g.n[x] : g.n_z, nu = x < 2 ? g.nu[x] : g.nu_z;
        if (M <= 0 || nu <= 0 || nu % M) return c->fail(TDSE_EINVAL, "nu must be a multiple of n");
        if (!fs_supported(M, nu / M)) return c->fail(TDSE_EUNSUPPORTED, "free space: n in 32..512, nu/n in {4,8,16}, nu <= 4096");
        if (!build_rule(F.ax[x], M, nu, p, g.gauss_q, g.n_r, g.H))
            return c->fail(TDSE_EINVAL, "contour rule: NE must exceed n/2 and the dense block 128 modes");
        F.ax[x].NT = 0;
        if (g.c_transform != TDSE_CT_DIRECT) {
            const int nt = choose_nt(F.ax[x]);
            if (g.c_transform == TDSE_CT_CHEBYSHEV && nt == 0)
                return c->fail(TDSE_EUNSUPPORTED, "C-type transforms: no Chebyshev interpolant of at most 64 terms "
                                                  "reaches FP64 rounding for this H");
            if (g.c_transform == TDSE_CT_CHEBYSHEV || (nt > 0 && nt < F.ax[x].NC)) F.ax[x].NT = nt;
        }
        F.NM *= (size_t)F.ax[x].N;
        F.NX *= (size_t)M;
    }
    // workspace
    const size_t B = c->B;
    size_t o = 0;
    auto take = [&](size_t bytes) { size_t r = o; o = align256(o + bytes); return r; };
    F.off = {};
    F.off.uhat = take(B * F.NM * 16);
    F.off.ring = take(B * c->RS * F.NM * c->rsz);
    F.off.chain_uhat = take((size_t)c->L * B * F.NM * 16);
    F.off.chain_ring = take((size_t)c->L * B * F.NM * c->rsz);
    F.off.chain_u = take((size_t)c->L * B * F.NX * 16);
    F.off.u = take(B * F.NX * 16);
    // 2D: Z [N0][M1]; 3D: Z [N0][N1][M2] and Y [N0][M1][M2]
    const size_t zel = c->d == 2 ? (size_t)F.ax[0].N * F.ax[1].M
                                 : (c->d == 3 ? (size_t)F.ax[0].N * F.ax[1].N * F.ax[2].M : 0);
    const size_t yel = c->d == 3 ? (size_t)F.ax[0].N * F.ax[1].M * F.ax[2].M : 0;
    F.off.Z = zel ? take(B * zel * c->rsz) : 0;
    F.off.Y = yel ? take(B * yel * c->rsz) : 0;
    const size_t vcopies = c->vshared ? 1 : B;
    F.off.V0 = take(vcopies * c->vrows * F.NX * 8);
    const size_t V0f = take(vcopies * c->vrows * F.NX * 8);
    F.off.tfac = take(B * (size_t)c->ntf * 8);
    F.off.phi = take(B * (size_t)c->d * c->ntf * 8);
    F.off.iv = take((size_t)c->n_int * sizeof(int2));
    for (int x = 0; x < c->d; ++x) {
        const FsAxisHost& A = F.ax[x];
        F.off.zeta[x] = take((size_t)A.N * 16);
        F.off.preI[x] = take((size_t)2 * A.NE * 16);
        F.off.postI[x] = take((size_t)2 * A.nu * 16);
        F.off.preF[x] = take((size_t)2 * A.nu * 16);
        F.off.postF[x] = take((size_t)2 * A.NE * 16);
        F.off.Gd[x] = take((size_t)A.ND * A.M * 16);
        F.off.Fd[x] = take((size_t)A.ND * A.M * 16);
        F.off.tw[x] = take((size_t)A.M * 16);
        F.off.P[x] = take(B * (size_t)c->n_int * A.N * 16);
        if (A.NT > 0) {
            F.off.Lf[x] = take((size_t)A.NT * A.M * 16);
            F.off.Li[x] = take((size_t)A.NT * A.M * 16);
            F.off.Tc[x] = take((size_t)A.NC * A.NT * 8);
            F.off.TcW[x] = take((size_t)A.NT * A.NC * 16);
            if (F.f32) {
                F.off.Lf_f[x] = take((size_t)A.NT * A.M * 8);
                F.off.Li_f[x] = take((size_t)A.NT * A.M * 8);
                F.off.Tc_f[x] = take((size_t)A.NC * A.NT * 4);
                F.off.TcW_f[x] = take((size_t)A.NT * A.NC * 8);
            }
        }
        if (F.f32) {
            F.off.preI_f[x] = take((size_t)2 * A.NE * 8);
            F.off.postI_f[x] = take((size_t)2 * A.nu * 8);
            F.off.preF_f[x] = take((size_t)2 * A.nu * 8);
            F.off.postF_f[x] = take((size_t)2 * A.NE * 8);
            F.off.Gd_f[x] = take((size_t)A.ND * A.M * 8);
            F.off.Fd_f[x] = take((size_t)A.ND * A.M * 8);
            F.off.tw_f[x] = take((size_t)A.M * 8);
            F.off.P_f[x] = take(B * (size_t)c->n_int * A.N * 8);
        }
    }
    size_t res_sums = 0, res_rho = 0, res_flags = 0, res_ncorr = 0;
    if (F.f32) {   // FP64 residual check of the FP32 step
        F.off.res_W = take(B * F.NM * 16);
        F.off.res_R = take(B * F.NM * 16);
        F.off.res_u = take(B * F.NX * 16);
        F.off.Z64 = zel ? take(B * zel * 16) : 0;
        F.off.Y64 = yel ? take(B * yel * 16) : 0;
        res_sums = take(B * 16);
        res_rho = take(B * 8);
        res_flags = take(B * 4);
        res_ncorr = take(B * 4);
    }
    F.off.scratch = take(256);
    F.off.end = o;
    c->ws_ckpt = o;
    F.off.g = take(B * sizeof(int));
    // not part of a checkpoint: exponents of the fixed-point tables; factor tables
    // of twice the lines for grids of more than 256 points
    for (int x = 0; x < c->d; ++x) {
        const FsAxisHost& A = F.ax[x];
        F.off.xj[x] = take((size_t)6 * A.M * sizeof(int));
        if (A.M <= 256) continue;
        F.off.postI[x] = take((size_t)4 * A.nu * 16);
        F.off.preF[x] = take((size_t)4 * A.nu * 16);
        if (F.f32) {
            F.off.postI_f[x] = take((size_t)4 * A.nu * 8);
            F.off.preF_f[x] = take((size_t)4 * A.nu * 8);
        }
    }
    c->ws_need = o;
    // fields the shared entry points use
    c->off = {};
    c->off.uhat = F.off.uhat;
    c->off.V0 = F.off.V0;
    c->off.V0f = V0f;
    c->off.tfac = F.off.tfac;
    c->off.phi = F.off.phi;
    c->off.iv = F.off.iv;
    c->off.scratch = F.off.scratch;
    c->off.res_sums = res_sums;
    c->off.res_rho = res_rho;
    c->off.res_flags = res_flags;
    c->off.res_ncorr = res_ncorr;
    return TDSE_OK;
}

namespace {
// Power of two that brings the modulus `big` into 1/2..1.
int exponent_of(double big) {
    int x = 0;
    if (big > 0.0) std::frexp(big, &x);
    return x;
}
// Fixed-point factors of complex values v, value i scaled by 2^-x(i).
template <class X>
std::vector<int4> factors(const std::vector<double>& v, X x) {
    std::vector<int4> w(v.size() / 2);
    for (size_t i = 0; i < w.size(); ++i) {
        fx_limbs(std::llround(std::ldexp(v[2 * i], 61 - x(i))), w[i].x, w[i].y);
        fx_limbs(std::llround(std::ldexp(v[2 * i + 1], 61 - x(i))), w[i].z, w[i].w);
    }
    return w;
}
}  // namespace

// The tables of every axis (functions of the configuration alone).
tdse_status fs_upload_tables(tdse_ctx* c, cudaStream_t s) {
    FsState& F = c->F;
    for (int x = 0; x < c->d; ++x) {
        FsAxisHost& A = F.ax[x];
        const AxisTables T = make_tables(A);
        const size_t M = A.M, R = A.M > 256 ? 2 * A.R : A.R;
        // largest modulus of entries first, first + step, .. of a table
        auto largest = [](const std::vector<double>& v, size_t first, size_t step, size_t n) {
            double big = 0.0;
            for (size_t i = 0; i < n; ++i)
                big = std::fmax(big, std::hypot(v[2 * (first + i * step)], v[2 * (first + i * step) + 1]));
            return big;
        };
        A.xI = exponent_of(largest(T.preI, 0, 1, T.preI.size() / 2));
        std::vector<int> xj(6 * M);
        for (size_t j = 0; j < M; ++j) {
            for (size_t b = 0; b < 2; ++b) {
                xj[b * M + j] = exponent_of(largest(T.preF, (b * M + j) * R, 1, R));
                xj[(3 + b) * M + j] = exponent_of(largest(T.postI, (b * M + j) * R, 1, R));
            }
            xj[2 * M + j] = exponent_of(std::fmax(largest(T.Fd, j, M, A.ND), A.NT ? largest(T.Lf, j, M, A.NT) : 0.0));
            xj[5 * M + j] = exponent_of(std::fmax(largest(T.Gd, j, M, A.ND), A.NT ? largest(T.Li, j, M, A.NT) : 0.0));
        }
        auto point = [&](int c) { return [&xj, M, c](size_t i) { return xj[c * M + i % M]; }; };     // [rows][M]
        auto lines = [&](int c) { return [&xj, R, M, c](size_t i) { return xj[c * M + i / R]; }; };  // [2][M][R], block 1 at c + 1
        auto whole = [](int x) { return [x](size_t) { return x; }; };
        auto up = [&](size_t off, const void* p, size_t bytes) -> cudaError_t {
            const cudaError_t e = cudaMemcpyAsync(c->P<char>(off), p, bytes, cudaMemcpyHostToDevice, s);
            return e != cudaSuccess ? e : cudaStreamSynchronize(s);   // the source is a temporary
        };
        auto up64 = [&](size_t off, const std::vector<double>& v) { return up(off, v.data(), v.size() * 8); };
        auto upfx = [&](size_t off, const std::vector<double>& v, auto e) {
            const std::vector<int4> w = factors(v, e);
            return up(off, w.data(), w.size() * sizeof(int4));
        };
        TDSE_CK(c, up64(F.off.zeta[x], T.zeta));
        TDSE_CK(c, up(F.off.xj[x], xj.data(), xj.size() * sizeof(int)));
        TDSE_CK(c, upfx(F.off.preI[x], T.preI, whole(A.xI)));
        TDSE_CK(c, upfx(F.off.postI[x], T.postI, lines(3)));
        TDSE_CK(c, upfx(F.off.preF[x], T.preF, lines(0)));
        TDSE_CK(c, upfx(F.off.postF[x], T.postF, whole(0)));
        TDSE_CK(c, upfx(F.off.Gd[x], T.Gd, point(5)));
        TDSE_CK(c, upfx(F.off.Fd[x], T.Fd, point(2)));
        TDSE_CK(c, upfx(F.off.tw[x], T.tw, whole(0)));
        if (A.NT > 0) {
            TDSE_CK(c, upfx(F.off.Lf[x], T.Lf, point(2)));
            TDSE_CK(c, upfx(F.off.Li[x], T.Li, point(5)));
            TDSE_CK(c, up64(F.off.Tc[x], T.Tc));
            TDSE_CK(c, up64(F.off.TcW[x], T.TcW));
        }
        // FP32 copies: each complex value rounded from the FP64 table
        auto up32 = [&](size_t off, const std::vector<double>& v) {
            const std::vector<float> t32(v.begin(), v.end());
            return up(off, t32.data(), t32.size() * 4);
        };
        if (F.f32) {
            TDSE_CK(c, up32(F.off.preI_f[x], T.preI));
            TDSE_CK(c, up32(F.off.postI_f[x], T.postI));
            TDSE_CK(c, up32(F.off.preF_f[x], T.preF));
            TDSE_CK(c, up32(F.off.postF_f[x], T.postF));
            TDSE_CK(c, up32(F.off.Gd_f[x], T.Gd));
            TDSE_CK(c, up32(F.off.Fd_f[x], T.Fd));
            TDSE_CK(c, up32(F.off.tw_f[x], T.tw));
            if (A.NT > 0) {
                TDSE_CK(c, up32(F.off.Lf_f[x], T.Lf));
                TDSE_CK(c, up32(F.off.Li_f[x], T.Li));
                TDSE_CK(c, up32(F.off.Tc_f[x], T.Tc));
                TDSE_CK(c, up32(F.off.TcW_f[x], T.TcW));
            }
        }
    }
    return TDSE_OK;
}

tdse_status fs_bind(tdse_ctx* c, cudaStream_t s) {
    c->F.g.assign(c->B, 0);
    TDSE_CK(c, cudaMemsetAsync(c->P<int>(c->F.off.g), 0, (size_t)c->B * sizeof(int), s));
    return fs_upload_tables(c, s);
}

// The one-step phase of an axis has modulus at most e^{H |dphi|}; over the
// history and all axes at most e^{7 H sum |dphi|}.  Its fixed-point factors
// hold moduli below 2^(1 + g), g < FS_WIDE; beyond that it is held in FP64: g of instances [lo, hi) for a field that changes
// by at most dphi per step (their phase tables are built after this, and take g
// to the device).
void fs_field_range(tdse_ctx* c, int lo, int hi, const double* dphi) {
    FsState& F = c->F;
    double growth = 0.0;
    for (int x = 0; x < c->d; ++x) growth += 7.0 * F.ax[x].H * std::fabs(dphi[x]);
    const double x = growth / M_LN2 - 1.0;
    const int g = x <= FS_WIDE - 1 ? std::max(0, (int)std::ceil(x)) : FS_WIDE;      // (a NaN: FS_WIDE)
    for (int b = lo; b < hi; ++b) F.g[b] = g;
}

// Largest change of phi per step and axis (the sum of the |changes| of its
// eighths), phi [d][ntf].
void fs_largest_dphi(const tdse_ctx* c, const double* phi, double* dphi) {
    for (int x = 0; x < c->d; ++x) {
        const double* p = phi + (size_t)x * c->ntf;
        for (int m = 0; m + SUB < c->ntf; m += SUB) {
            double t = 0.0;
            for (int i = 0; i < SUB; ++i) t += std::fabs(p[m + i + 1] - p[m + i]);
            dphi[x] = std::fmax(dphi[x], t);
        }
    }
}

// After a checkpoint is loaded: the range of its fields, from its flags (two
// bytes per instance, g + 1 above bit 0 of the first) or, where they have none,
// from its phi tables.
tdse_status fs_loaded_field_range(tdse_ctx* c, const char* flags, cudaStream_t s) {
    FsState& F = c->F;
    std::vector<double> phi((size_t)c->d * c->ntf);
    for (int b = 0; b < c->B; ++b) {
        const int g = (unsigned char)flags[2 * b] >> 1;
        double dphi[3] = {0.0, 0.0, 0.0};
        if (!g) {
            TDSE_CK(c, cudaMemcpyAsync(phi.data(), c->P<double>(F.off.phi) + (size_t)b * phi.size(), phi.size() * 8,
                                       cudaMemcpyDeviceToHost, s));
            TDSE_CK(c, cudaStreamSynchronize(s));
            fs_largest_dphi(c, phi.data(), dphi);
        }
        fs_field_range(c, b, b + 1, dphi);
        if (g) F.g[b] = std::min(g - 1, FS_WIDE);
    }
    return TDSE_OK;
}

tdse_status fs_build_phase_tables(tdse_ctx* c, int b, cudaStream_t s) {
    const FsState& F = c->F;
    const int2* iv = c->P<int2>(F.off.iv);
    for (int x = 0; x < c->d; ++x) {
        const FsAxisHost& A = F.ax[x];
        const size_t at = (size_t)b * c->n_int * A.N;
        const double* phi = c->P<double>(F.off.phi) + ((size_t)b * c->d + x) * c->ntf;
        TDSE_CK(c, launch_fs_phase(c->P<int4>(F.off.P[x]) + at, F.f32 ? c->P<float2>(F.off.P_f[x]) + at : nullptr,
                                   c->P<int>(F.off.g) + b, F.g[b], c->P<double2>(F.off.zeta[x]), A.N, iv, c->n_int, phi, c->cfg.dt, s));
    }
    return TDSE_OK;
}

tdse_status fs_set_initial(tdse_ctx* c, int b, const double* u0, cudaMemcpyKind kind, cudaStream_t s) {
    const FsState& F = c->F;
    TDSE_CK(c, cudaMemcpyAsync(c->P<double2>(F.off.u) + (size_t)b * F.NX, u0, F.NX * 16, kind, s));
    return TDSE_OK;
}

tdse_status fs_steps(tdse_ctx* c, int nsteps, cudaStream_t s) {
    if (!c->inited) {
        tdse_status st = fs_init(c, s);
        if (st != TDSE_OK) return st;
    }
    int k = 0;
    while (k < nsteps) {
        const int n = c->step + 1;
        if (n <= c->S) {
            tdse_status st = fs_startup_step(c, n, s);
            if (st != TDSE_OK) return st;
            c->step = n;
            ++k;
            continue;
        }
        int run_len = nsteps - k;
        const bool check = c->F.f32 && c->res_every > 0;
        if (check) {   // stop at the next step to check
            const int to_check = c->res_every - c->step % c->res_every;
            if (to_check < run_len) run_len = to_check;
        }
        tdse_status st = fs_adams(c, c->step, run_len, s);
        if (st != TDSE_OK) return st;
        c->step += run_len;
        k += run_len;
        if (check && c->step % c->res_every == 0) {
            st = fs_residual_check(c, s);
            if (st != TDSE_OK) return st;
        }
    }
    return TDSE_OK;
}

tdse_status fs_read_u(tdse_ctx* c, int lo, int hi, double* out, cudaMemcpyKind kind, cudaStream_t s) {
    const FsState& F = c->F;
    TDSE_CK(c, cudaMemcpyAsync(out, c->P<double2>(F.off.u) + (size_t)lo * F.NX, (size_t)(hi - lo) * F.NX * 16, kind,
                               s));
    return TDSE_OK;
}

extern "C" tdse_status tdse_free_rule(const tdse_ctx* c, int axis, int* N, double* zeta, double* w) {
    if (!c || !N || !c->fs || axis < 0 || axis >= c->d) return TDSE_EINVAL;
    const FsAxisHost& A = c->F.ax[axis];
    *N = A.N;
    if (zeta) std::memcpy(zeta, A.zeta.data(), A.zeta.size() * 8);
    if (w) std::memcpy(w, A.w.data(), A.w.size() * 8);
    return TDSE_OK;
}

extern "C" tdse_status tdse_free_choose_H_prec(double eps, double vnorm, double phimax, int dim, int precision,
                                               double* H_out) {
    if (!H_out || dim < 1 || dim > 3 || !(eps > 0.0) || !(vnorm >= 0.0) || !(phimax >= 0.0)) return TDSE_EINVAL;
    if (precision != TDSE_FP64 && precision != TDSE_MIXED) return TDSE_EINVAL;
    // machine epsilon of the arithmetic that evaluates the contour sums
    const double eps_m = std::ldexp(1.0, precision == TDSE_FP64 ? -52 : -23);
    const double H = std::log(eps / ((1.0 + vnorm) * eps_m)) / (2.0 * dim * (1.0 + phimax));
    if (!(H > 0.0) || !std::isfinite(H)) return TDSE_EINVAL;
    *H_out = H;
    return TDSE_OK;
}

extern "C" tdse_status tdse_free_choose_H(double eps, double vnorm, double phimax, int dim, double* H_out) {
    return tdse_free_choose_H_prec(eps, vnorm, phimax, dim, TDSE_FP64, H_out);
}

extern "C" int tdse_free_cheb_terms(const tdse_ctx* c, int axis) {
    if (!c || !c->fs || axis < 0 || axis >= c->d) return -1;
    return c->F.ax[axis].NT;
}
