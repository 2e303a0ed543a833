// init.cuh -- the initial state from (drho, u, grad u), un-streamed into the buffer.
//
// f = f_eq(drho, rho0 u) + T^-1 m_neq - Fbar/2 at each node, with the first-order viscous moments
// m_neq of the given gradient (D3Q19: eq. (YuLuobasis); D2Q9 and D3Q15: the same first-order
// Chapman-Enskog moments worked out on their bases), from FP64 inputs.
//
// Opposite-pair form: with cj = c.j, cF = c.F, g0 = drho - 1.5 j.(j - F)/rho0 and e = (T^-1 m_neq)_a
// (m_neq holds even moments only, so both velocities of a pair get the same e),
//   E = w g0 + 4.5 w cj (cj - cF)/rho0 + e,  O = 1.5 w (2 cj - cF),  f_a = E + O,  f_b = E - O.
//
// What bounds it: 180 B a node with a gradient (FP32), and the arithmetic.  In FP64 a population-
// by-population form takes about 530 FP64 operations a node on the pipe that finishes 2 a clock and SM:
// 5.9 ms for a 192^3 FP32 box with a gradient against 0.35 ms in this form (its bytes take 0.19 ms at the measured copy
// bandwidth; the error against 64 bits is 2.5e-8 either way).  FP64 storage runs the pair form above in FP64; the other
// storages run it in pairs of floats (dfloat.cuh: 48 bits, rounded once to FP32 at the end, as the FP64 result was), and
// only nodes next to a moving wall, with a result that is not finite or with values near the smallest of FP32
// repeat it in FP64.
#pragma once

#include "dfloat.cuh"
#include "step.cuh"

namespace lbm {

// arithmetic type of the initialiser: FP64 for FP64 storage, float pairs otherwise
template <class ST>
using InitX = typename std::conditional<std::is_same<ST, double>::value, double, DF>::type;

template <class X>
struct XC;
template <>
struct XC<double> {
    __host__ __device__ static constexpr double c(double v) { return v; }
    static __device__ __forceinline__ double in(double v) { return v; }
    static __device__ __forceinline__ double root(double v) { return sqrt(v); }
    static __device__ __forceinline__ double full(double v) { return v; }
    template <class R>
    static __device__ __forceinline__ R out(double v) {
        return R(v);
    }
};
template <>
struct XC<DF> {
    __host__ __device__ static constexpr DF c(double v) { return DF(float(v), float(v - double(float(v)))); }
    static __device__ __forceinline__ DF in(double v) { return DF(v); }
    static __device__ __forceinline__ DF in(float v) { return DF(v); }
    static __device__ __forceinline__ DF root(DF v) { return df_sqrt(v); }
    static __device__ __forceinline__ double full(DF v) { return df_double(v); }
    template <class R>
    static __device__ __forceinline__ R out(DF v) {
        return R(df_value(v));
    }
};

template <class X>
struct InitConst {
    int closure;
    X r0, ir0, ir15, ir45;    // rho0, 1/rho0, 1.5/rho0, 4.5/rho0
    X tau0, smag, e1;         // 1/s_nu of the rates, 3 Cs^2/rho0, m_neq,1 / (|T_1|^2 div j)
    X F[3];
};

template <class L, class X>
inline InitConst<X> init_const(const StepArgs<double>& a, int closure) {
    InitConst<X> k;
    k.closure = closure;
    k.r0 = XC<X>::c(a.rho0);
    k.ir0 = XC<X>::c(a.inv_rho0);
    k.ir15 = XC<X>::c(1.5 * a.inv_rho0);
    k.ir45 = XC<X>::c(4.5 * a.inv_rho0);
    k.tau0 = XC<X>::c(a.tau0);
    k.smag = XC<X>::c(a.smag_c3 * a.inv_rho0);
    const double m1 = L::Q == 19 ? -38.0 / (3.0 * a.s[1]) : (L::Q == 15 ? -2.0 / (3.0 * a.s[1]) : -2.0 / a.s[1]);
    k.e1 = XC<X>::c(m1 / norm2<L>(1));
    for (int d = 0; d < 3; ++d) k.F[d] = XC<X>::c(a.F[d]);
    return k;
}

// the closure's tau at the prescribed gradient G = rho0 grad u (explicit, since S is given)
template <class L, class X>
__device__ __forceinline__ X init_tau(const StepArgs<double>& a, const InitConst<X>& k, const X (&G)[3][3]) {
    if (k.closure == CL_NEWTON) return k.tau0;
    X e[3], tr = X(0.0f);
    sfor<L::D>([&](auto d) { e[d] = G[CV(d)][CV(d)]; });
    if (k.closure == CL_SMAG_DEV) {  // traceless part only
        sfor<L::D>([&](auto d) { tr = tr + e[d]; });
        tr = tr * XC<X>::c(1.0 / L::D);
        sfor<L::D>([&](auto d) { e[d] = e[d] - tr; });
    }
    X ss = X(0.0f), sh = X(0.0f);
    sfor<L::D>([&](auto d) { ss = fma(e[d], e[d], ss); });
    sfor<L::NS>([&](auto c) {
        constexpr int p = strain_axis<L>(CV(c), 0), q = strain_axis<L>(CV(c), 1);
        if constexpr (p != q) {
            const X g = G[p][q] + G[q][p];
            sh = fma(g, g, sh);
        }
    });
    const X n2 = X(2.0f) * ss + sh, n = XC<X>::root(n2);  // |rho0 S|, |S| = sqrt(2 S:S)
    if (k.closure == CL_POWERLAW) {
        // a pair whose squares left the FP32 range, or lost bits below it (tau follows log |S| down to any strain, and
        // only gradients that are zero give zero): no clamp may hide it, the node is redone in FP64
        if constexpr (!std::is_same<X, double>::value) {
            float g = 0.0f;
            sfor<L::D>([&](auto p) { sfor<L::D>([&](auto q) { g = fmaxf(g, fabsf(G[CV(p)][CV(q)].h)); }); });
            if (!(XC<X>::full(n) <= 3.0e38) || (n2.h < 0x1p-100f && g > 0.0f)) return X(nanf(""));
        }
        double t = 0.5 + a.pl_k3 * pow(XC<X>::full(n) * a.inv_rho0, a.pl_nm1);
        if (!(t >= a.pl_tau_min)) t = a.pl_tau_min;
        if (t > a.pl_tau_max) t = a.pl_tau_max;
        return XC<X>::in(t);
    }
    return fma(k.smag, n, k.tau0);
}

// even part e of T^-1 m_neq per pair (e0: rest) for the gradient G = rho0 grad u
template <class L, class X>
__device__ __forceinline__ void init_noneq(const InitConst<X>& k, X tau, const X (&G)[3][3], X& e0, X (&e)[L::NP]) {
    X div = G[0][0] + G[1][1];
    if constexpr (L::D == 3) div = div + G[2][2];
    const X t3 = tau * XC<X>::c(-1.0 / 3.0);
    X D[L::Q];
    sfor<L::Q>([&](auto i) { D[i] = X(0.0f); });
    auto shear = [&](int p, int q, int m) { return t3 * XC<X>::c(1.0 / m) * (G[p][q] + G[q][p]); };
    if constexpr (L::D == 3) {
        constexpr int ww = L::Q == 19 ? 11 : 10, xy = L::Q == 19 ? 13 : 11;
        D[9] = t3 * XC<X>::c(2.0 / norm2<L>(9)) * (X(3.0f) * G[0][0] - div);
        D[ww] = t3 * XC<X>::c(2.0 / norm2<L>(ww)) * (G[1][1] - G[2][2]);
        D[xy] = shear(0, 1, norm2<L>(xy));
        D[xy + 1] = shear(1, 2, norm2<L>(xy + 1));
        D[xy + 2] = shear(0, 2, norm2<L>(xy + 2));
    } else {
        D[7] = t3 * XC<X>::c(2.0 / norm2<L>(7)) * (G[0][0] - G[1][1]);
        D[8] = shear(0, 1, norm2<L>(8));
    }
    Xf<L>::viscous_even(D, e);
    const X m1 = k.e1 * div;
    e0 = X(float(L::T(1, 0))) * m1;  // the viscous rows of T have no rest entry
    constexpr int ax = L::pa(0), dg = L::pa(L::NP - 1);
    const X ma = X(float(L::T(1, ax))) * m1, md = X(float(L::T(1, dg))) * m1;  // axis, diagonal pairs
    sfor<L::NP>([&](auto p) {
        constexpr int i = L::pa(CV(p));
        constexpr bool axis = L::wnum(i) == L::wnum(ax);
        e[p] = e[p] + (axis ? ma : md);
    });
}

// the node's populations
template <class L, bool FORCE, class X, class R>
__device__ __forceinline__ void init_node(const InitConst<X>& k, X dr, const X (&j)[3], const X (&F)[3], bool neq,
                                          const X (&G)[3][3], X tau, R (&f)[L::Q]) {
    X e0 = X(0.0f), e[L::NP];
    sfor<L::NP>([&](auto p) { e[p] = X(0.0f); });
    if (neq) init_noneq<L>(k, tau, G, e0, e);
    X g = X(0.0f);
    sfor<L::D>([&](auto d) {
        if constexpr (FORCE)
            g = fma(j[d], j[d] - F[d], g);
        else
            g = fma(j[d], j[d], g);
    });
    const X g0 = dr - k.ir15 * g;
    constexpr int ax = L::pa(0), dg = L::pa(L::NP - 1);
    constexpr double w0 = double(L::wnum(0)) / L::WDEN;
    constexpr double wa = double(L::wnum(ax)) / L::WDEN, wd = double(L::wnum(dg)) / L::WDEN;
    f[0] = XC<X>::template out<R>(fma(XC<X>::c(w0), g0, e0));
    const X ga = XC<X>::c(wa) * g0, gd = XC<X>::c(wd) * g0;
    const X qa = XC<X>::c(wa) * k.ir45, qd = XC<X>::c(wd) * k.ir45;
    sfor<L::NP>([&](auto p) {
        constexpr int i = L::pa(CV(p));
        constexpr bool axis = L::wnum(i) == L::wnum(ax);
        X cj = X(0.0f), cF = X(0.0f);
        bool first = true;
        sfor<L::D>([&](auto d) {
            constexpr int c = L::c(i, CV(d));
            if constexpr (c != 0) {
                cj = first ? (c > 0 ? j[d] : -j[d]) : (c > 0 ? cj + j[d] : cj - j[d]);
                if constexpr (FORCE) cF = first ? (c > 0 ? F[d] : -F[d]) : (c > 0 ? cF + F[d] : cF - F[d]);
                first = false;
            }
        });
        const X t = FORCE ? cj - cF : cj;
        const X E = (fma((axis ? qa : qd) * cj, t, e[p])) + (axis ? ga : gd);
        const X O = FORCE ? XC<X>::c(1.5 * (axis ? wa : wd)) * (cj + t) : XC<X>::c(3.0 * (axis ? wa : wd)) * cj;
        f[L::pa(CV(p))] = XC<X>::template out<R>(E + O);
        f[L::pb(CV(p))] = XC<X>::template out<R>(E - O);
    });
}

// un-stream: write each population where the pull of (node, i) will read it.  Nodes with no wall next
// to them write at node - c_i, wrapped by index; the others by the boundary rules.
template <class L, class ST, class V>
__device__ __forceinline__ void unstream(const StepArgs<double>& a, int x, int y, int z, const V (&f)[L::Q]) {
    using R = typename Store<ST>::R;
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const int node = (z * ny + y) * nx + x;
    ST* __restrict__ buf = static_cast<ST*>(a.dst);
    if (no_wall_next<L, ST>(a, x, y, z)) {
        const WrapYZ w(y, z, nx, ny, nz);
        const int dxm = x == 0 ? nx - 1 : -1, dxp = x == nx - 1 ? 1 - nx : 1;
        sfor<L::Q>([&](auto i) {
            constexpr int cx = L::c(CV(i), 0), cy = L::c(CV(i), 1), cz = L::c(CV(i), 2);
            const int to = node + (cx > 0 ? dxm : (cx < 0 ? dxp : 0)) + w.template off<cy, cz>();
            Store<ST>::st(buf + CV(i) * a.stride + to, R(f[i]));
        });
        return;
    }
    const int dims[3] = {nx, ny, nz};
    const int pos[3] = {x, y, z};
    sfor<L::Q>([&](auto i) {
        int s[3];
        int nout = 0, face = -1;
        sfor<3>([&](auto ax) {
            constexpr int c = L::c(CV(i), CV(ax));
            s[ax] = pos[ax] - c;
            if constexpr (c != 0) {
                if (s[ax] < 0 || s[ax] >= dims[ax]) {
                    const int fc = 2 * CV(ax) + (s[ax] < 0 ? 0 : 1);
                    if ((a.wall_mask >> fc) & 1) {
                        ++nout;
                        face = fc;
                    } else {
                        s[ax] = s[ax] < 0 ? s[ax] + dims[ax] : s[ax] - dims[ax];
                    }
                }
            }
        });
        if (nout == 0) {
            Store<ST>::st(buf + CV(i) * a.stride + (s[2] * ny + s[1]) * nx + s[0], R(f[i]));
        } else {
            V v = f[i];
            if (nout == 1 && ((a.lid_mask >> face) & 1)) {
                const double cu = L::c(CV(i), 0) * a.lid[face][0] + L::c(CV(i), 1) * a.lid[face][1] +
                                  L::c(CV(i), 2) * a.lid[face][2];
                v = V(double(v) - 6.0 * (double(L::wnum(CV(i))) / L::WDEN) * a.rho0 * cu);
            }
            Store<ST>::st(buf + opp<L>(CV(i)) * a.stride + node, R(v));
        }
    });
}

// One node in arithmetic X: loads, populations, tau; returns whether X holds every result (in FP64
// always true: its infinities and NaN are the result).
template <class L, class ST, bool FORCE, class X, class V>
__device__ __forceinline__ bool init_at(const StepArgs<double>& a, const InitConst<X>& k, int node,
                                        const double* __restrict__ drho, const double* __restrict__ u,
                                        const double* __restrict__ gu,
                                        const typename Store<ST>::R* __restrict__ ffield,
                                        V (&f)[L::Q], V& tau_out) {
    const long long N = (long long)a.nx * a.ny * a.nz;  // component offsets (up to 8N) exceed 2^31 on big grids
    // every load first: the conversions branch, and a load behind a branch waits for it (192^3, with the blocks
    // cut at row ends that left a quarter of the threads idle: 0.60 ms)
    double du[3] = {0.0, 0.0, 0.0}, dg[9];
    typename Store<ST>::R dF[3];
    const double dd = drho[node];
    sfor<L::D>([&](auto d) { du[d] = u[CV(d) * N + node]; });
    if (gu) sfor<L::D * L::D>([&](auto c) { dg[c] = gu[CV(c) * N + node]; });
    if constexpr (FORCE) {
        if (ffield) sfor<L::D>([&](auto d) { dF[d] = ffield[CV(d) * N + node]; });
    }
    X j[3], F[3], G[3][3];
    sfor<3>([&](auto d) {
        F[d] = k.F[CV(d)];
        sfor<3>([&](auto e) { G[CV(d)][CV(e)] = X(0.0f); });
    });
    sfor<L::D>([&](auto d) {
        j[d] = k.r0 * XC<X>::in(du[d]);
        if constexpr (FORCE) {
            if (ffield) F[d] = XC<X>::in(dF[d]);
        }
    });
    const X dr = XC<X>::in(dd);
    if (gu)
        sfor<L::D>([&](auto p) {
            sfor<L::D>([&](auto q) { G[CV(p)][CV(q)] = k.r0 * XC<X>::in(dg[CV(p) * L::D + CV(q)]); });
        });
    const X tau = init_tau<L>(a, k, G);
    tau_out = XC<X>::template out<V>(tau);
    init_node<L, FORCE>(k, dr, j, F, gu != nullptr, G, tau, f);
    if constexpr (std::is_same<X, double>::value) return true;
    V s = V(0);
    sfor<L::Q>([&](auto i) { s += r_abs(f[i]); });
    // false for NaN too; below 2^-90 a pair's low part, 2^-24 to 2^-48 of the value, comes near the smallest FP32
    // numbers and loses bits
    return s + tau_out < V(3.0e38f) && (s >= V(0x1p-90f) || s == V(0));
}

// the node in FP64 up to the stores: float pairs that left the FP32 range on the way, at either end, and nodes next to
// a moving wall, whose term joins the population before it is rounded
template <class L, class ST, bool FORCE>
__device__ __noinline__ void init_again(const StepArgs<double>& a, const InitConst<double>& k, int x, int y, int z,
                                        const double* drho, const double* u, const double* gu,
                                        const typename Store<ST>::R* ffield, typename Store<ST>::R* tau_field) {
    const int node = (z * a.ny + y) * a.nx + x;
    double f[L::Q], tau;
    init_at<L, ST, FORCE, double>(a, k, node, drho, u, gu, ffield, f, tau);
    if (tau_field) tau_field[node] = typename Store<ST>::R(tau);
    unstream<L, ST>(a, x, y, z, f);
}

template <class L, class ST, bool FORCE>
__global__ void __launch_bounds__(128) k_init(const StepArgs<double> a, const InitConst<InitX<ST>> k,
                                              const InitConst<double> kd, const NodeMap g,
                                              const double* __restrict__ drho,
                                              const double* __restrict__ u, const double* __restrict__ gu,
                                              const typename Store<ST>::R* __restrict__ ffield,
                                              typename Store<ST>::R* __restrict__ tau_field) {
    using R = typename Store<ST>::R;
    int x, y, z;
    if (!node_in_order<1>(a, g, x, y, z)) return;
    const int node = (z * a.ny + y) * a.nx + x;
    R f[L::Q], tau;
    bool ok = init_at<L, ST, FORCE>(a, k, node, drho, u, gu, ffield, f, tau);
    if constexpr (!std::is_same<R, double>::value)
        ok = ok && (a.lid_mask == 0 || no_wall_next<L, ST>(a, x, y, z));
    if (!ok) {
        init_again<L, ST, FORCE>(a, kd, x, y, z, drho, u, gu, ffield, tau_field);
        return;
    }
    if (tau_field) tau_field[node] = tau;  // the lagged closure keeps it as the tau of the first step
    unstream<L, ST>(a, x, y, z, f);
}

}  // namespace lbm
