// step.cuh -- the fused MRT lattice Boltzmann step.
//
// A step pulls each node's 19 (or 9) pre-collision populations from the previous post-collision
// buffer (f_i(x) = f*_i(x - c_i), Sec. 2 eq. (mrteq)), forms S by Yu's formula (eq. (LuoS)) or
// Chai's formula (eq. (ChaiS)), solves the strain-rate closure for tau, relaxes in moment space
// (eq. (mrteqvT)) with the discrete force, and stores f* at the node: a single pass over HBM,
// 2 q values per node.
//
// Both routes write the collision in "delta form", f* = f - (increment), so that the
// storage-precision rounding acts only on the small collision increment:
//   Yu route:   D_k = (s_k mneq_k - TF_k) / |T_k|^2 over moments k, mneq = T f - m_eq + TF/2,
//               f*_i = f_i - sum_k T_ki D_k.
//   Chai route: fneq_i = f_i - f_eq_i + Fbar_i/2, mneq = T fneq;  S = -sum_i c_i c_i Omega_i / (2 rho0 cs^2)
//               of Omega = T^-1 L mneq, whose contraction with c c is folded into T^-1 at compile time
//               (chai_contract);  f* as on the Yu route.
// TF = T Fbar is the moment vector of the Guo-type discrete force Fbar_i =
// w_i[(c_i - u).F/cs^2 + (c_i.u)(c_i.F)/cs^4]; it equals the j-derivative of m_eq along F.
// With a closure the viscous rates are unknown, so both routes split S = A + s_nu B (exact:
// S is linear in the rates) and solve the scalar fixed point for tau = 1/s_nu.
//
// A thread owns one node (this file), or with 16-bit storage two x-adjacent nodes that share the
// pull's address arithmetic and collide side by side in packed FP32-pair arithmetic
// (step_pair.cuh, which forms f* from the post-collision moments instead of in delta form).
//
// All lattice coefficients enter as compile-time constants: loops over populations and moments
// are compile-time sequences (sfor) so each entry of T and c folds into an add, a subtract or
// an FMA with an immediate.  Accumulators start at -0.0, the exact additive identity, so the
// first term needs no special case.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include <type_traits>
#include <utility>

#include "lattice.cuh"
#include "launch.h"
#include "power_law.h"


namespace lbm {

enum { CL_NEWTON = 0, CL_SMAG = 1, CL_POWERLAW = 2, CL_SMAG_LAGGED = 3, CL_SMAG_DEV = 4 };
enum { F_YU = 0, F_CHAI = 1 };

// ------------------------------------------------------------------------------------------
// compile-time loops

template <class F, int... Is>
__host__ __device__ __forceinline__ void sfor_impl(F&& f, std::integer_sequence<int, Is...>) {
    (f(std::integral_constant<int, Is>{}), ...);
}
template <int N, class F>
__host__ __device__ __forceinline__ void sfor(F&& f) {
    sfor_impl(f, std::make_integer_sequence<int, N>{});
}
#define CV(x) (decltype(x)::value)

// fused multiply-add under one name for both compute types
__device__ __forceinline__ float fma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma(double a, double b, double c) { return ::fma(a, b, c); }

// the pulled populations of two x-adjacent nodes (lo: the even node, hi: the odd one)
struct F2 {
    float2 v;
    F2() = default;
    __device__ __forceinline__ F2(float a, float b) : v{a, b} {}
    __device__ __forceinline__ explicit F2(float2 u) : v(u) {}
    __device__ __forceinline__ float lo() const { return v.x; }
    __device__ __forceinline__ float hi() const { return v.y; }
};

// acc + t x for a compile-time integer t
template <int T, class R>
__device__ __forceinline__ R cadd(R acc, R x) {
    if constexpr (T == 0)
        return acc;
    else if constexpr (T == 1)
        return acc + x;
    else if constexpr (T == -1)
        return acc - x;
    else
        return fma(R(float(T)), x, acc);
}
template <class R>
__device__ __forceinline__ constexpr R nzero() {
    return R(-0.0f);
}
// a constant given in double, rounded once to the compute type (exact for the FP64 path)
template <class R>
__device__ __forceinline__ constexpr R cst(double c) {
    if constexpr (std::is_same<R, double>::value)
        return c;
    else
        return R(float(c));
}

// ------------------------------------------------------------------------------------------
// storage types: scalar access, and the pair load of the two-node path.  ld/ld2 read through
// the non-coherent path (the buffer is read-only for the whole kernel); ldc/ld2c read through L2
// only (ld.global.cg), for a kernel that reads populations other blocks of the same kernel wrote
// after synchronising with them.

template <class ST>
struct Store;
template <>
struct Store<double> {
    using R = double;
    static __device__ __forceinline__ R ld(const double* p) { return __ldg(p); }
    static __device__ __forceinline__ R ldc(const double* p) { return __ldcg(p); }
    static __device__ __forceinline__ void st(double* p, R v) { __stcs(p, v); }
};
template <>
struct Store<float> {
    using R = float;
    static __device__ __forceinline__ R ld(const float* p) { return __ldg(p); }
    static __device__ __forceinline__ R ldc(const float* p) { return __ldcg(p); }
    static __device__ __forceinline__ void st(float* p, R v) { __stcs(p, v); }
    // aligned pair p[0], p[1] (p 8-byte aligned)
    static __device__ __forceinline__ F2 ld2(const float* p) { return F2(__ldg(reinterpret_cast<const float2*>(p))); }
    static __device__ __forceinline__ F2 ld2c(const float* p) { return F2(__ldcg(reinterpret_cast<const float2*>(p))); }
};
template <>
struct Store<__half> {
    using R = float;
    static __device__ __forceinline__ R ld(const __half* p) { return __half2float(__ldg(p)); }
    static __device__ __forceinline__ R ldc(const __half* p) { return __half2float(__ldcg(p)); }
    static __device__ __forceinline__ void st(__half* p, R v) { *p = __float2half_rn(v); }
    // aligned pair p[0] = lo, p[1] = hi (p 4-byte aligned), each rounded to nearest as st does
    static __device__ __forceinline__ void st2(__half* p, R lo, R hi) {
        *reinterpret_cast<__half2*>(p) = __floats2half2_rn(lo, hi);
    }
    static __device__ __forceinline__ F2 ld2(const __half* p) {
        return F2(__half22float2(__ldg(reinterpret_cast<const __half2*>(p))));
    }
    static __device__ __forceinline__ F2 ld2c(const __half* p) {
        return F2(__half22float2(__ldcg(reinterpret_cast<const __half2*>(p))));
    }
};
template <>
struct Store<__nv_bfloat16> {
    using R = float;
    static __device__ __forceinline__ R ld(const __nv_bfloat16* p) { return __bfloat162float(__ldg(p)); }
    static __device__ __forceinline__ R ldc(const __nv_bfloat16* p) { return __bfloat162float(__ldcg(p)); }
    static __device__ __forceinline__ void st(__nv_bfloat16* p, R v) { *p = __float2bfloat16_rn(v); }
    static __device__ __forceinline__ void st2(__nv_bfloat16* p, R lo, R hi) {
        *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(lo, hi);
    }
    static __device__ __forceinline__ F2 ld2(const __nv_bfloat16* p) {
        return F2(__bfloat1622float2(__ldg(reinterpret_cast<const __nv_bfloat162*>(p))));
    }
    static __device__ __forceinline__ F2 ld2c(const __nv_bfloat16* p) {
        return F2(__bfloat1622float2(__ldcg(reinterpret_cast<const __nv_bfloat162*>(p))));
    }
};

__device__ __forceinline__ float r_abs(float x) { return fabsf(x); }
__device__ __forceinline__ double r_abs(double x) { return fabs(x); }
// Closure arithmetic: in FP32 the approximate reciprocal, reciprocal square root, logarithm and power of
// two (errors of a few ulp, far inside the FP32 tolerance of S), in FP64 the IEEE operations.  The reciprocal and the
// square root are the instructions that take subnormals as zero, without the scaling around them (channel
// 256x128x128, 20 steps, Smagorinsky, GLUPS with the scaling / without: FP16 Yu 61.1 / 64.1, FP32 Chai 41.7 / 42.1):
// tau lies above 1/2, and a strain under 1.1e-19, whose square is subnormal, adds less than half a last place to
// a tau0 of 1/2 and more for any 3 Cs^2 below 2.7e11.  So is the power of two: |S|^(n-1) is never subnormal for n up
// to 2.69, nor seen beside 1/2 beyond that unless 3K is above 2^100.  The logarithm is not: tau of the power
// law follows log |S| down to any strain.
__device__ __forceinline__ float c_rcp(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ double c_rcp(double x) { return 1.0 / x; }
__device__ __forceinline__ float c_sqrt(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return x >= 1.17549435e-38f ? x * y : 0.0f;
}
__device__ __forceinline__ double c_sqrt(double x) { return sqrt(x); }
__device__ __forceinline__ float c_log2(float x) { return __log2f(x); }
__device__ __forceinline__ float c_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// |S|^(n-1) of the power-law closure from q2 = 2 S:S = |S|^2: in FP32 one fast power of q2 with
// exponent (n-1)/2 (no square root; exactly 1 for n = 1; a q2 rounded below zero counts as zero,
// as the square root's guard does), in FP64 the IEEE square root and power.
__device__ __forceinline__ float strain_pow(float q2, float nm1) {
    return nm1 == 0.0f ? 1.0f : c_exp2(0.5f * nm1 * c_log2(fmaxf(q2, 0.0f)));
}
__device__ __forceinline__ double strain_pow(double q2, double nm1) { return pow(sqrt(q2), nm1); }

// ------------------------------------------------------------------------------------------
// kernel arguments (by value; scalar type RS = float or double)

template <class RS>
struct StepArgs {
    int nx, ny, nz;
    int z0, nzc;           // planes computed: [z0, z0 + nzc) (all, or the owned planes between halo planes)
    long long stride;      // elements between population arrays
    const void* src;       // post-collision buffer of the previous step
    void* dst;             // post-collision buffer of this step
    const void* srcp[19];  // src + i * stride, population i (filled on the host)
    void* dstp[19];        // dst + i * stride
    const RS* force_field; // d x N, or nullptr for the uniform force F
    RS F[3];
    RS s[19];              // relaxation rates; the viscous entries hold 1/tau0
    RS skn[19];            // s_k / |T_k|^2
    RS rho0, inv_rho0, tau0;
    RS smag_c3;            // 3 Cs^2
    RS pl_k3, pl_nm1, pl_tau_min, pl_tau_max, pl_tol;  // 3K, n-1, clamp, tolerance
    PowerLawGuess pl_guess;  // first guess of tau
    int smag_iters, pl_max_iter;
    int wall_mask;         // bit f: face f is not periodic (wall or lid)
    int lid_mask;          // bit f: face f is a moving wall
    RS lid[6][3];
    RS* S_out;
    RS* tau_out;
    RS* drho_out;
    RS* u_out;
    RS* tau_field;         // lagged closure: N stored taus, read and rewritten in place by each node
};

// ------------------------------------------------------------------------------------------
// lattice-derived compile-time facts

template <class L>
__host__ __device__ constexpr int opp(int i) {
    for (int p = 0; p < L::NP; ++p) {
        if (L::pa(p) == i) return L::pb(p);
        if (L::pb(p) == i) return L::pa(p);
    }
    return i;
}

// strain components: xx, yy, zz, xy, yz, xz (3D) or xx, yy, xy (2D)
template <class L>
__host__ __device__ constexpr int strain_axis(int cpt, int which) {
    constexpr int ab3[6][2] = {{0, 0}, {1, 1}, {2, 2}, {0, 1}, {1, 2}, {0, 2}};
    constexpr int ab2[3][2] = {{0, 0}, {1, 1}, {0, 1}};
    return L::NS == 6 ? ab3[cpt][which] : ab2[cpt][which];
}

// ------------------------------------------------------------------------------------------
// moment transforms

// m_K = sum_i T_Ki f_i from the rest population and the opposite-pair sums P / differences Dd
template <class L, int K, class R>
__device__ __forceinline__ R moment(R f0, const R (&P)[L::NP], const R (&Dd)[L::NP]) {
    R acc = nzero<R>();
    if constexpr (even_moment<L>(K)) {
        acc = cadd<L::T(K, 0)>(acc, f0);
        sfor<L::NP>([&](auto p) { acc = cadd<L::T(K, L::pa(CV(p)))>(acc, P[p]); });
    } else {
        sfor<L::NP>([&](auto p) { acc = cadd<L::T(K, L::pa(CV(p)))>(acc, Dd[p]); });
    }
    return acc;
}

// out_i = sum_k T_ki D_k over the moments k whose bit is set in USE, via even and odd parts of
// each opposite pair
template <class L, uint32_t USE, class R>
__device__ __forceinline__ void back_transform(const R (&D)[L::Q], R (&out)[L::Q]) {
    R r = nzero<R>();
    sfor<L::Q>([&](auto k) {
        if constexpr ((USE >> CV(k)) & 1u) r = cadd<L::T(CV(k), 0)>(r, D[k]);
    });
    out[0] = r;
    sfor<L::NP>([&](auto p) {
        constexpr int a = L::pa(CV(p)), b = L::pb(CV(p));
        R E = nzero<R>(), O = nzero<R>();
        sfor<L::Q>([&](auto k) {
            if constexpr ((USE >> CV(k)) & 1u) {
                if constexpr (even_moment<L>(CV(k)))
                    E = cadd<L::T(CV(k), a)>(E, D[k]);
                else
                    O = cadd<L::T(CV(k), a)>(O, D[k]);
            }
        });
        out[a] = E + O;
        out[b] = E - O;
    });
}

// out_a = out_b = E_p for the opposite pairs p = (a, b) of out_i = sum_k T_ki D_k over the viscous
// moments, which are all even (the rest population gets nothing: their rows have no rest entry)
template <class L, class R>
__device__ __forceinline__ void viscous_pairs(const R (&D)[L::Q], R (&E)[L::NP]) {
    sfor<L::NP>([&](auto p) {
        R e = nzero<R>();
        sfor<L::Q>([&](auto k) {
            if constexpr (L::viscous(CV(k))) e = cadd<L::T(CV(k), L::pa(CV(p)))>(e, D[k]);
        });
        E[p] = e;
    });
}

template <class L>
__host__ __device__ constexpr uint32_t mask_nonconserved() {
    uint32_t m = 0;
    for (int k = 0; k < L::Q; ++k)
        if (!L::conserved(k)) m |= 1u << k;
    return m;
}
template <class L>
__host__ __device__ constexpr uint32_t mask_all_but_density() {
    return ((1u << L::Q) - 1u) & ~1u;
}
template <class L>
__host__ __device__ constexpr uint32_t mask_all() {
    return (1u << L::Q) - 1u;
}

// Forward and backward transforms.  The generic form (any lattice) sums the nonzero entries of
// each row of T over the opposite-pair sums and differences.  D3Q19 and D3Q15 have hand-factored forms
// that share partial sums (axis / edge / corner butterflies) between rows; they compute the same maps.
template <class L>
struct Xf {
    // m[k] = (T f)_k for every k (m[0] = drho, m[3], m[5], m[7] = raw momentum)
    template <class R>
    static __device__ __forceinline__ void forward(R f0, const R (&P)[L::NP], const R (&Dd)[L::NP], R (&m)[L::Q]) {
        sfor<L::Q>([&](auto k) { m[k] = moment<L, CV(k)>(f0, P, Dd); });
    }
    template <uint32_t USE, class R>
    static __device__ __forceinline__ void backward(const R (&D)[L::Q], R (&out)[L::Q]) {
        back_transform<L, USE>(D, out);
    }
    template <class R>
    static __device__ __forceinline__ void viscous_even(const R (&D)[L::Q], R (&E)[L::NP]) {
        viscous_pairs<L>(D, E);
    }
};

template <>
struct Xf<D3Q19> {
    // pair order: x (1,2), y (3,4), z (5,6), (7,10), (8,9), (11,14), (12,13), (15,18), (16,17)

    // viscous_pairs from shared partial sums (moments 9, 11, 13, 14, 15)
    template <class R>
    static __device__ __forceinline__ void viscous_even(const R (&a)[19], R (&E)[9]) {
        const R p = a[9] + a[11], m = a[9] - a[11], t = R(-2.0f) * a[9];
        E[0] = R(2.0f) * a[9];
        E[1] = -m;
        E[2] = -p;
        E[3] = p + a[13];
        E[4] = p - a[13];
        E[5] = m + a[15];
        E[6] = m - a[15];
        E[7] = t + a[14];
        E[8] = t - a[14];
    }

    // Even and odd parts of out_i = sum_k T_ki a_k over the non-conserved moments that are not viscous (1, 2, 4, 6,
    // 8, 10, 12, 16, 17, 18): E0 for the rest population, E_p + O_p and E_p - O_p for pair p
    template <class R>
    static __device__ __forceinline__ void fixed_pairs(const R (&a)[19], R& E0, R (&E)[9], R (&O)[9]) {
        E0 = fma(R(12.0f), a[2], R(-30.0f) * a[1]);
        const R B1 = fma(R(-4.0f), a[2], R(-11.0f) * a[1]);  // axis pairs
        const R B2 = fma(R(8.0f), a[1], a[2]);               // edge pairs
        const R s = a[10] + a[12], t = a[10] - a[12];
        E[0] = fma(R(-4.0f), a[10], B1);
        E[1] = fma(R(2.0f), t, B1);
        E[2] = fma(R(2.0f), s, B1);
        E[3] = E[4] = B2 + s;
        E[5] = E[6] = B2 + t;
        E[7] = E[8] = fma(R(-2.0f), a[10], B2);
        O[0] = R(-4.0f) * a[4];
        O[1] = R(-4.0f) * a[6];
        O[2] = R(-4.0f) * a[8];
        const R u1 = a[4] + a[16], v1 = a[6] - a[17];
        O[3] = v1 + u1;
        O[4] = v1 - u1;
        const R u2 = a[4] - a[16], v2 = a[8] + a[18];
        O[5] = v2 + u2;
        O[6] = v2 - u2;
        const R u3 = a[6] + a[17], v3 = a[8] - a[18];
        O[7] = v3 + u3;
        O[8] = v3 - u3;
    }

    template <class R>
    static __device__ __forceinline__ void forward(R f0, const R (&P)[9], const R (&D)[9], R (&m)[19]) {
        const R Exy = P[3] + P[4], Exz = P[5] + P[6], Eyz = P[7] + P[8];
        const R Pyz = P[1] + P[2];
        const R Sax = P[0] + Pyz;
        const R Q = Exy + Exz;
        const R Sed = Q + Eyz;
        m[0] = f0 + Sax + Sed;
        const R Ex = (D[3] - D[4]) + (D[5] - D[6]);
        const R Ey = (D[3] + D[4]) + (D[7] - D[8]);
        const R Ez = (D[5] + D[6]) + (D[7] + D[8]);
        m[3] = D[0] + Ex;
        m[5] = D[1] + Ey;
        m[7] = D[2] + Ez;
        m[4] = fma(R(-4.0f), D[0], Ex);
        m[6] = fma(R(-4.0f), D[1], Ey);
        m[8] = fma(R(-4.0f), D[2], Ez);
        m[1] = fma(R(8.0f), Sed, fma(R(-11.0f), Sax, R(-30.0f) * f0));
        m[2] = fma(R(-4.0f), Sax, fma(R(12.0f), f0, Sed));
        const R Qm = fma(R(-2.0f), Eyz, Q);
        m[9] = fma(R(2.0f), P[0], Qm - Pyz);
        m[10] = fma(R(-4.0f), P[0], fma(R(2.0f), Pyz, Qm));
        const R dyz = P[1] - P[2], dxyz = Exy - Exz;
        m[11] = dyz + dxyz;
        m[12] = fma(R(-2.0f), dyz, dxyz);
        m[13] = P[3] - P[4];
        m[14] = P[7] - P[8];
        m[15] = P[5] - P[6];
        m[16] = (D[3] - D[4]) - (D[5] - D[6]);
        m[17] = (D[7] - D[8]) - (D[3] + D[4]);
        m[18] = (D[5] + D[6]) - (D[7] + D[8]);
    }

    // out_i = sum_k T_ki a_k.  The factored form needs every non-conserved a_k; with CONS the
    // momentum entries a_3, a_5, a_7 are included too (a_0 is always absent).  Other masks use
    // the generic form.
    template <uint32_t USE, class R>
    static __device__ __forceinline__ void backward(const R (&a)[19], R (&out)[19]) {
        constexpr uint32_t NC = mask_nonconserved<D3Q19>();
        if constexpr (USE != NC && USE != mask_all_but_density<D3Q19>() && USE != mask_all<D3Q19>()) {
            back_transform<D3Q19, USE>(a, out);
        } else {
            constexpr bool CONS = (USE >> 3) & 1u, DENS = USE & 1u;  // T_0i = 1 for every i
            out[0] = DENS ? fma(R(12.0f), a[2], fma(R(-30.0f), a[1], a[0])) : fma(R(12.0f), a[2], R(-30.0f) * a[1]);
            // axis populations
            const R B1 = DENS ? fma(R(-4.0f), a[2], fma(R(-11.0f), a[1], a[0])) : fma(R(-4.0f), a[2], R(-11.0f) * a[1]);
            const R C = fma(R(2.0f), a[10], -a[9]);
            const R W = fma(R(-2.0f), a[12], a[11]);
            const R Ex = fma(R(-2.0f), C, B1);
            const R BC = B1 + C;
            const R Ey = BC + W;
            const R Ez = BC - W;
            R Ox, Oy, Oz;
            if constexpr (CONS) {
                Ox = fma(R(-4.0f), a[4], a[3]);
                Oy = fma(R(-4.0f), a[6], a[5]);
                Oz = fma(R(-4.0f), a[8], a[7]);
            } else {
                Ox = R(-4.0f) * a[4];
                Oy = R(-4.0f) * a[6];
                Oz = R(-4.0f) * a[8];
            }
            out[1] = Ex + Ox;
            out[2] = Ex - Ox;
            out[3] = Ey + Oy;
            out[4] = Ey - Oy;
            out[5] = Ez + Oz;
            out[6] = Ez - Oz;
            // edge populations
            const R B2 = DENS ? fma(R(8.0f), a[1], a[2] + a[0]) : fma(R(8.0f), a[1], a[2]);
            const R G = a[9] + a[10], H = a[11] + a[12];
            R X = a[4], Y = a[6], Z = a[8];
            if constexpr (CONS) {
                X += a[3];
                Y += a[5];
                Z += a[7];
            }
            const R BG = B2 + G;
            {  // xy edges: (7,10) and (8,9)
                const R base = BG + H;
                const R E4 = base + a[13], E5 = base - a[13];
                const R u = X + a[16], v = Y - a[17];
                const R O4 = v + u, O5 = v - u;
                out[7] = E4 + O4;
                out[10] = E4 - O4;
                out[8] = E5 + O5;
                out[9] = E5 - O5;
            }
            {  // xz edges: (11,14) and (12,13)
                const R base = BG - H;
                const R E6 = base + a[15], E7 = base - a[15];
                const R u = X - a[16], v = Z + a[18];
                const R O6 = v + u, O7 = v - u;
                out[11] = E6 + O6;
                out[14] = E6 - O6;
                out[12] = E7 + O7;
                out[13] = E7 - O7;
            }
            {  // yz edges: (15,18) and (16,17)
                const R base = fma(R(-2.0f), G, B2);
                const R E8 = base + a[14], E9 = base - a[14];
                const R u = Y + a[17], v = Z - a[18];
                const R O8 = v + u, O9 = v - u;
                out[15] = E8 + O8;
                out[18] = E8 - O8;
                out[16] = E9 + O9;
                out[17] = E9 - O9;
            }
        }
    }
};

template <>
struct Xf<D3Q15> {
    // pair order: x (1,2), y (3,4), z (5,6), corners (7,14), (8,13), (9,12), (10,11); the four corner
    // pairs are combined by two-level butterflies shared between rows
    template <class R>
    static __device__ __forceinline__ void forward(R f0, const R (&P)[7], const R (&D)[7], R (&m)[15]) {
        const R a = P[3] + P[6], b = P[4] + P[5], c = P[3] - P[6], d = P[4] - P[5];
        const R Sc = a + b, Sax = P[0] + (P[1] + P[2]);
        const R u = D[3] + D[5], v = D[4] + D[6], w = D[3] - D[5], x = D[4] - D[6];
        const R Cx = u - v, Cy = w + x, Cz = u + v;
        m[0] = f0 + Sax + Sc;
        m[1] = fma(R(-2.0f), f0, Sc - Sax);
        m[2] = fma(R(16.0f), f0, fma(R(-4.0f), Sax, Sc));
        m[3] = D[0] + Cx;
        m[4] = fma(R(-4.0f), D[0], Cx);
        m[5] = D[1] + Cy;
        m[6] = fma(R(-4.0f), D[1], Cy);
        m[7] = D[2] + Cz;
        m[8] = fma(R(-4.0f), D[2], Cz);
        m[9] = fma(R(3.0f), P[0], -Sax);
        m[10] = P[1] - P[2];
        m[11] = a - b;
        m[12] = c + d;
        m[13] = c - d;
        m[14] = w - x;
    }

    // fixed_pairs of D3Q19 on this basis (moments 1, 2, 4, 6, 8, 14)
    template <class R>
    static __device__ __forceinline__ void fixed_pairs(const R (&a)[15], R& E0, R (&E)[7], R (&O)[7]) {
        E0 = fma(R(16.0f), a[2], R(-2.0f) * a[1]);
        E[0] = E[1] = E[2] = fma(R(-4.0f), a[2], -a[1]);
        E[3] = E[4] = E[5] = E[6] = a[1] + a[2];
        O[0] = R(-4.0f) * a[4];
        O[1] = R(-4.0f) * a[6];
        O[2] = R(-4.0f) * a[8];
        const R p = a[8] + a[6], m = a[8] - a[6], c = a[4] + a[14], d = a[4] - a[14];
        O[3] = p + c;
        O[4] = p - c;
        O[5] = m + d;
        O[6] = m - d;
    }

    // viscous_pairs from shared partial sums (moments 9..13)
    template <class R>
    static __device__ __forceinline__ void viscous_even(const R (&a)[15], R (&E)[7]) {
        E[0] = R(2.0f) * a[9];
        E[1] = a[10] - a[9];
        E[2] = -(a[9] + a[10]);
        const R s1 = a[11] + a[13], s2 = a[11] - a[13];
        E[3] = a[12] + s1;
        E[4] = a[12] - s1;
        E[5] = -(a[12] + s2);
        E[6] = s2 - a[12];
    }

    // out_i = sum_k T_ki a_k for every non-conserved a_k (with CONS also a_3, a_5, a_7); other
    // masks use the generic form
    template <uint32_t USE, class R>
    static __device__ __forceinline__ void backward(const R (&a)[15], R (&out)[15]) {
        constexpr uint32_t NC = mask_nonconserved<D3Q15>();
        if constexpr (USE != NC && USE != mask_all_but_density<D3Q15>() && USE != mask_all<D3Q15>()) {
            back_transform<D3Q15, USE>(a, out);
        } else {
            constexpr bool CONS = (USE >> 3) & 1u, DENS = USE & 1u;  // T_0i = 1 for every i
            out[0] = DENS ? fma(R(16.0f), a[2], fma(R(-2.0f), a[1], a[0])) : fma(R(16.0f), a[2], R(-2.0f) * a[1]);
            // axis populations
            const R B1 = DENS ? fma(R(-4.0f), a[2], a[0] - a[1]) : fma(R(-4.0f), a[2], -a[1]);
            const R Ex = fma(R(2.0f), a[9], B1), BC = B1 - a[9];
            const R Ey = BC + a[10], Ez = BC - a[10];
            R Ox, Oy, Oz, X = a[4], Y = a[6], Z = a[8];
            if constexpr (CONS) {
                Ox = fma(R(-4.0f), a[4], a[3]);
                Oy = fma(R(-4.0f), a[6], a[5]);
                Oz = fma(R(-4.0f), a[8], a[7]);
                X += a[3];
                Y += a[5];
                Z += a[7];
            } else {
                Ox = R(-4.0f) * a[4];
                Oy = R(-4.0f) * a[6];
                Oz = R(-4.0f) * a[8];
            }
            out[1] = Ex + Ox;
            out[2] = Ex - Ox;
            out[3] = Ey + Oy;
            out[4] = Ey - Oy;
            out[5] = Ez + Oz;
            out[6] = Ez - Oz;
            // corner populations: even parts B2 +- a11 +- a12 +- a13, odd parts +-X +-Y +-Z +- a14
            const R B2 = DENS ? (a[1] + a[2]) + a[0] : a[1] + a[2];
            const R s = B2 + a[11], t = B2 - a[11], g = a[12] + a[13], h = a[12] - a[13];
            const R U = Z + Y, V = Z - Y, p = X + a[14], r = a[14] - X;
            const R E3 = s + g, E6 = s - g, E4 = t + h, E5 = t - h;
            const R O3 = U + p, O4 = U - p, O5 = V - r, O6 = V + r;
            out[7] = E3 + O3;
            out[14] = E3 - O3;
            out[8] = E4 + O4;
            out[13] = E4 - O4;
            out[9] = E5 + O5;
            out[12] = E5 - O5;
            out[10] = E6 + O6;
            out[11] = E6 - O6;
        }
    }
};

// sum_i c_ia c_ib T_ki for the strain component cpt = (a, b)
template <class L>
__host__ __device__ constexpr int second_moment(int cpt, int k) {
    int s = 0;
    for (int i = 0; i < L::Q; ++i)
        s += L::c(i, strain_axis<L>(cpt, 0)) * L::c(i, strain_axis<L>(cpt, 1)) * L::T(k, i);
    return s;
}

// Chai's formula, S = kS sum_i c_i c_i (T^-1 L mn)_i with kS = -1/(2 rho0 cs^2), for the moments mn = T f_neq
// of the non-equilibrium distributions.  The contraction and T^-1 = T^t diag(1/|T_k|^2) are both
// constant, so their product is formed at compile time: S_c = kS sum_k (sum_i c_i c_i T_ki) D_k with
// D_k = s_k mn_k / |T_k|^2, in which only the energy moment and the viscous moments have nonzero sums.
// Forming T^-1 L mn in the q directions and contracting it there, as the formula is written (omega_split), made the
// FP32 step one of instructions and registers: D3Q19 channel 256x128x128, 20 steps, 39.1 GLUPS against 41.7.
template <class L, class R, class Take>
__device__ __forceinline__ void chai_contract(const R (&D)[L::Q], R kS, Take take, R (&S)[L::NS]) {
    sfor<L::NS>([&](auto cpt) {
        R acc = nzero<R>();
        sfor<L::Q>([&](auto k) {
            if constexpr (take(CV(k))) acc = cadd<second_moment<L>(CV(cpt), CV(k))>(acc, D[k]);
        });
        S[cpt] = kS * acc;
    });
}

// The same formula as it is written, for S = A + s_nu B: Omega = T^-1 L mn of the rate-independent moments (by pairs
// Ef0, Ef, Of) and of the viscous ones (Ev; both velocities of a pair get the same), contracted with c c, to
// which odd parts add nothing.  Lattices with a closure and 16-bit storage step by this one: the folded product
// rounds S differently in its last FP32 place, and where that moves a population across a rounding
// boundary of the storage the neighbours follow, until after some 20 steps the states are a storage
// rounding apart everywhere (D3Q15 BF16 channel 256x128x128: 5e-3 of the state, which is also how far
// either is from 64 bits).  The off-diagonal rate-independent sums cancel exactly (the two edge or four corner pairs
// involved hold the same value), and the factor 2 of a pair's two velocities is exact in kS2 = 2 kS.
template <class L, int CPT, class R>
__device__ __forceinline__ R contract_pairs(const R (&E)[L::NP]) {
    constexpr int a = strain_axis<L>(CPT, 0), b = strain_axis<L>(CPT, 1);
    R acc = nzero<R>();
    sfor<L::NP>([&](auto p) { acc = cadd<L::c(L::pa(CV(p)), a) * L::c(L::pa(CV(p)), b)>(acc, E[p]); });
    return acc;
}
template <class L, class RS, class R>
__device__ __forceinline__ void omega_split(const StepArgs<RS>& a, const R (&mn)[L::Q], R ir0, R& Ef0, R (&Ef)[L::NP],
                                            R (&Of)[L::NP], R (&Ev)[L::NP], R (&A)[L::NS], R (&B)[L::NS]) {
    const R kS2 = R(-3.0f) * ir0;
    R D[L::Q];
    sfor<L::Q>([&](auto k) {
        if constexpr (L::viscous(CV(k)))
            D[k] = cst<R>(1.0 / norm2<L>(CV(k))) * mn[k];
        else if constexpr (!L::conserved(CV(k)))
            D[k] = R(a.skn[k]) * mn[k];
    });
    Xf<L>::fixed_pairs(D, Ef0, Ef, Of);
    Xf<L>::viscous_even(D, Ev);
    sfor<L::NS>([&](auto c) {
        if constexpr (CV(c) < L::D)
            A[c] = kS2 * contract_pairs<L, CV(c)>(Ef);
        else
            A[c] = R(0.0f);
        B[c] = kS2 * contract_pairs<L, CV(c)>(Ev);
    });
}
// S:T of a diagonal S
template <class L, class R>
__device__ __forceinline__ R diag_dot(const R (&S)[L::NS], const R (&T)[L::NS]) {
    if constexpr (L::NS == 6)
        return fma(S[0], T[0], fma(S[1], T[1], S[2] * T[2]));
    else
        return fma(S[0], T[0], S[1] * T[1]);
}

// ------------------------------------------------------------------------------------------
// equilibrium moments (closed form) and force moments TF = d m_eq / d j . F, both written with
// u = j / rho0 formed once

template <class L>
struct Eq;

template <>
struct Eq<D3Q19> {
    // eq. (meq): w_eps = 3, w_epsj = -11/2, w_xx = -1/2
    template <class R>
    static __device__ __forceinline__ void meq(R drho, const R (&j)[3], const R (&u)[3], R (&m)[19]) {
        const R ju = fma(j[0], u[0], fma(j[1], u[1], j[2] * u[2]));
        m[0] = drho;
        m[1] = fma(R(19.0f), ju, R(-11.0f) * drho);
        m[2] = fma(R(-5.5f), ju, R(3.0f) * drho);
        m[3] = j[0];
        m[4] = cst<R>(-2.0 / 3.0) * j[0];
        m[5] = j[1];
        m[6] = cst<R>(-2.0 / 3.0) * j[1];
        m[7] = j[2];
        m[8] = cst<R>(-2.0 / 3.0) * j[2];
        m[9] = fma(R(3.0f) * j[0], u[0], -ju);
        m[10] = R(-0.5f) * m[9];
        m[11] = fma(j[1], u[1], -(j[2] * u[2]));
        m[12] = R(-0.5f) * m[11];
        m[13] = j[0] * u[1];
        m[14] = j[1] * u[2];
        m[15] = j[0] * u[2];
        m[16] = R(0.0f);
        m[17] = R(0.0f);
        m[18] = R(0.0f);
    }
    template <class R>
    static __device__ __forceinline__ void tforce(const R (&u)[3], const R (&F)[3], R (&t)[19]) {
        const R uF = fma(u[0], F[0], fma(u[1], F[1], u[2] * F[2]));
        t[0] = R(0.0f);
        t[1] = R(38.0f) * uF;
        t[2] = R(-11.0f) * uF;
        t[3] = F[0];
        t[4] = cst<R>(-2.0 / 3.0) * F[0];
        t[5] = F[1];
        t[6] = cst<R>(-2.0 / 3.0) * F[1];
        t[7] = F[2];
        t[8] = cst<R>(-2.0 / 3.0) * F[2];
        t[9] = fma(R(6.0f) * u[0], F[0], R(-2.0f) * uF);
        t[10] = R(-0.5f) * t[9];
        t[11] = R(2.0f) * fma(u[1], F[1], -(u[2] * F[2]));
        t[12] = R(-0.5f) * t[11];
        t[13] = fma(u[0], F[1], u[1] * F[0]);
        t[14] = fma(u[1], F[2], u[2] * F[1]);
        t[15] = fma(u[0], F[2], u[2] * F[0]);
        t[16] = R(0.0f);
        t[17] = R(0.0f);
        t[18] = R(0.0f);
    }
    // moments with identically zero equilibrium and force parts (ghost moments t_x, t_y, t_z)
    static __host__ __device__ constexpr bool ghost(int k) { return k >= 16; }
    // Yu formula eq. (LuoS) split as S = A + s_nu B (A: the s1 m1 part); c1 = s1/(38 rho0), ir0 = 1/rho0
    template <class R>
    static __device__ __forceinline__ void yu_split(const R (&mn)[19], R c1, R ir0, R (&A)[6], R (&B)[6]) {
        const R a = -(c1 * mn[1]);
        A[0] = a;
        A[1] = a;
        A[2] = a;
        A[3] = R(0.0f);
        A[4] = R(0.0f);
        A[5] = R(0.0f);
        const R h = R(0.25f) * ir0;
        const R k = R(-1.5f) * ir0;
        B[0] = (R(-0.5f) * ir0) * mn[9];
        B[1] = h * fma(R(-3.0f), mn[11], mn[9]);
        B[2] = h * fma(R(3.0f), mn[11], mn[9]);
        B[3] = k * mn[13];
        B[4] = k * mn[14];
        B[5] = k * mn[15];
    }
    static constexpr double YU_A = 1.0 / 38.0;  // c1 = s1 * YU_A / rho0
};

template <>
struct Eq<D3Q15> {
    // T f_eq of the He-Luo equilibrium on the d'Humieres D3Q15 basis
    template <class R>
    static __device__ __forceinline__ void meq(R drho, const R (&j)[3], const R (&u)[3], R (&m)[15]) {
        const R ju = fma(j[0], u[0], fma(j[1], u[1], j[2] * u[2]));
        m[0] = drho;
        m[1] = ju - drho;
        m[2] = fma(R(-5.0f), ju, drho);
        m[3] = j[0];
        m[4] = cst<R>(-7.0 / 3.0) * j[0];
        m[5] = j[1];
        m[6] = cst<R>(-7.0 / 3.0) * j[1];
        m[7] = j[2];
        m[8] = cst<R>(-7.0 / 3.0) * j[2];
        m[9] = fma(R(3.0f) * j[0], u[0], -ju);
        m[10] = fma(j[1], u[1], -(j[2] * u[2]));
        m[11] = j[0] * u[1];
        m[12] = j[1] * u[2];
        m[13] = j[0] * u[2];
        m[14] = R(0.0f);
    }
    template <class R>
    static __device__ __forceinline__ void tforce(const R (&u)[3], const R (&F)[3], R (&t)[15]) {
        const R uF = fma(u[0], F[0], fma(u[1], F[1], u[2] * F[2]));
        t[0] = R(0.0f);
        t[1] = R(2.0f) * uF;
        t[2] = R(-10.0f) * uF;
        t[3] = F[0];
        t[4] = cst<R>(-7.0 / 3.0) * F[0];
        t[5] = F[1];
        t[6] = cst<R>(-7.0 / 3.0) * F[1];
        t[7] = F[2];
        t[8] = cst<R>(-7.0 / 3.0) * F[2];
        t[9] = fma(R(6.0f) * u[0], F[0], R(-2.0f) * uF);
        t[10] = R(2.0f) * fma(u[1], F[1], -(u[2] * F[2]));
        t[11] = fma(u[0], F[1], u[1] * F[0]);
        t[12] = fma(u[1], F[2], u[2] * F[1]);
        t[13] = fma(u[0], F[2], u[2] * F[0]);
        t[14] = R(0.0f);
    }
    // m_xyz has zero equilibrium and force parts
    static __host__ __device__ constexpr bool ghost(int k) { return k == 14; }
    // Yu-type D3Q15 formula (Sec. 5.4 procedure): S_xx = -(s_e m_e + s_nu m_3pxx)/(2 rho0),
    // S_yy,zz = -(2 s_e m_e - s_nu m_3pxx +- 3 s_nu m_pww)/(4 rho0), S_ab = -3 s_nu m_pab/(2 rho0);
    // c1 = s_e/(2 rho0)
    template <class R>
    static __device__ __forceinline__ void yu_split(const R (&mn)[15], R c1, R ir0, R (&A)[6], R (&B)[6]) {
        const R a = -(c1 * mn[1]);
        A[0] = a;
        A[1] = a;
        A[2] = a;
        A[3] = R(0.0f);
        A[4] = R(0.0f);
        A[5] = R(0.0f);
        const R h = R(0.25f) * ir0;
        const R k = R(-1.5f) * ir0;
        B[0] = (R(-0.5f) * ir0) * mn[9];
        B[1] = h * fma(R(-3.0f), mn[10], mn[9]);
        B[2] = h * fma(R(3.0f), mn[10], mn[9]);
        B[3] = k * mn[11];
        B[4] = k * mn[12];
        B[5] = k * mn[13];
    }
    static constexpr double YU_A = 1.0 / 2.0;
};

template <>
struct Eq<D2Q9> {
    template <class R>
    static __device__ __forceinline__ void meq(R drho, const R (&j)[3], const R (&u)[3], R (&m)[9]) {
        const R ju = fma(j[0], u[0], j[1] * u[1]);
        m[0] = drho;
        m[1] = fma(R(3.0f), ju, R(-2.0f) * drho);
        m[2] = fma(R(-3.0f), ju, drho);
        m[3] = j[0];
        m[4] = -j[0];
        m[5] = j[1];
        m[6] = -j[1];
        m[7] = fma(j[0], u[0], -(j[1] * u[1]));
        m[8] = j[0] * u[1];
    }
    template <class R>
    static __device__ __forceinline__ void tforce(const R (&u)[3], const R (&F)[3], R (&t)[9]) {
        const R uF = fma(u[0], F[0], u[1] * F[1]);
        t[0] = R(0.0f);
        t[1] = R(6.0f) * uF;
        t[2] = R(-6.0f) * uF;
        t[3] = F[0];
        t[4] = -F[0];
        t[5] = F[1];
        t[6] = -F[1];
        t[7] = R(2.0f) * fma(u[0], F[0], -(u[1] * F[1]));
        t[8] = fma(u[0], F[1], u[1] * F[0]);
    }
    static __host__ __device__ constexpr bool ghost(int) { return false; }
    // Yu-type D2Q9 formula (Sec. 5.4 procedure): S_xx,yy = -(s_e m_e +- 3 s_nu m_pxx)/(4 rho0),
    // S_xy = -3 s_nu m_pxy / (2 rho0);  c1 = s_e/(4 rho0)
    template <class R>
    static __device__ __forceinline__ void yu_split(const R (&mn)[9], R c1, R ir0, R (&A)[3], R (&B)[3]) {
        const R a = -(c1 * mn[1]);
        A[0] = a;
        A[1] = a;
        A[2] = R(0.0f);
        const R h = R(0.75f) * ir0;
        B[0] = -(h * mn[7]);
        B[1] = h * mn[7];
        B[2] = (R(-1.5f) * ir0) * mn[8];
    }
    static constexpr double YU_A = 1.0 / 4.0;
};

// Chai route: the effective non-equilibrium distributions f - f_eq + Fbar/2 of the He-Luo
// equilibrium (eq. (edf)) and the Guo-type force, in opposite-pair form, formed directly.  With
// cj = c.j, cu = c.u, cF = c.F (c = c_a of pair p, weight w), g = u.(j - F) and
// B = 2 drho - 3 g, f_eq_a + f_eq_b = 2w (drho + 4.5 cj cu - 1.5 j.u), f_eq_a - f_eq_b = 6 w cj,
// Fbar_a + Fbar_b = 2w (9 cu cF - 3 u.F), Fbar_a - Fbar_b = 6 w cF, Fbar_0 = -3 w0 u.F, so that
//   (f_eq - Fbar/2)_a + (f_eq - Fbar/2)_b = w B + 9 w cu (cj - cF),
//   (f_eq - Fbar/2)_a - (f_eq - Fbar/2)_b = 3 w (2 cj - cF),
//   (f_eq - Fbar/2)_0 = w0 B / 2.
// Pn_p = P_p - (first), Dn_p = D_p - (second), fn0 = f0 - (third).
template <class L, bool FORCE, class R>
__device__ __forceinline__ void noneq_pairs(R f0, const R (&P)[L::NP], const R (&Dd)[L::NP], R drho, const R (&j)[3],
                                            const R (&u)[3], const R (&F)[3], R& fn0, R (&Pn)[L::NP],
                                            R (&Dn)[L::NP]) {
    R g = fma(j[0], u[0], fma(j[1], u[1], j[2] * u[2]));
    if constexpr (FORCE) g = fma(-u[0], F[0], fma(-u[1], F[1], fma(-u[2], F[2], g)));
    const R B = fma(R(-3.0f), g, R(2.0f) * drho);
    constexpr double w0 = double(L::wnum(0)) / L::WDEN;
    fn0 = fma(cst<R>(-0.5 * w0), B, f0);
    sfor<L::NP>([&](auto p) {
        constexpr int i = L::pa(CV(p));
        constexpr int cx = L::c(i, 0), cy = L::c(i, 1), cz = L::c(i, 2);
        constexpr double w = double(L::wnum(i)) / L::WDEN;
        const R cj = cadd<cz>(cadd<cy>(cadd<cx>(nzero<R>(), j[0]), j[1]), j[2]);
        const R cu = cadd<cz>(cadd<cy>(cadd<cx>(nzero<R>(), u[0]), u[1]), u[2]);
        R t = cj, t2 = R(2.0f) * cj;
        if constexpr (FORCE) {
            const R cF = cadd<cz>(cadd<cy>(cadd<cx>(nzero<R>(), F[0]), F[1]), F[2]);
            t = cj - cF;
            t2 = fma(R(2.0f), cj, -cF);
        }
        Pn[p] = fma(cst<R>(-9.0 * w) * cu, t, fma(cst<R>(-w), B, P[p]));
        Dn[p] = fma(cst<R>(-3.0 * w), t2, Dd[p]);
    });
}

// ------------------------------------------------------------------------------------------
// closure: solve tau with S = A + (1/tau) B

template <class L, class R>
__device__ __forceinline__ R strain_dot(const R (&S)[L::NS], const R (&T)[L::NS]) {
    // S:T with the off-diagonal components counted twice
    if constexpr (L::NS == 6)
        return fma(S[0], T[0], fma(S[1], T[1], S[2] * T[2])) +
               R(2.0f) * fma(S[3], T[3], fma(S[4], T[4], S[5] * T[5]));
    else
        return fma(S[0], T[0], S[1] * T[1]) + R(2.0f) * (S[2] * T[2]);
}

template <class L, class R>
__device__ __forceinline__ void affine(const R (&A)[L::NS], const R (&B)[L::NS], R s, R (&S)[L::NS]) {
#pragma unroll
    for (int c = 0; c < L::NS; ++c) S[c] = fma(s, B[c], A[c]);
}

// First guess of the power law's tau (power_law.h): its root when the rate-free part of S vanishes.
template <class RS>
__device__ __forceinline__ RS power_law_start(RS qc, const StepArgs<RS>& a) {
    const PowerLawGuess& g = a.pl_guess;
    const float x = fmaf(g.ax, c_log2(2.0f * float(qc)), g.x0);
    if (!(x > -1.0f)) return a.pl_tau_min;
    if (x >= 1.0f) return a.pl_tau_max;
    float v = g.p[POWER_LAW_DEGREE];
    sfor<POWER_LAW_DEGREE>([&](auto i) { v = fmaf(v, x, g.p[POWER_LAW_DEGREE - 1 - CV(i)]); });
    return RS(0.5f + c_exp2(v));
}

// tau at one node from the quadratic |S|^2 = 2 (qa + qb2 s + qc s^2), s = 1/tau (qa = A:A,
// qb2 = 2 A:B, qc = B:B: exact since S = A + s B), as the fixed point of the closure's map F.
// Smagorinsky: `smag_iters` sweeps from tau0, stopping early only when a sweep returns its input bit
// for bit (every later sweep would too).  Power law: F(tau) = 1/2 + 3K |S|^(n-1), clamped, until
// |F(tau) - tau| <= pl_tol F(tau) or pl_max_iter sweeps.  With a guess (the contractive range of n, see
// power_law.h) the sweeps start from it and one that stays inside the clamps is followed by a Newton
// step; there F has one fixed point, so the stopping rule accepts the same one.  A sweep costs 20
// instructions and 3 special-function ones, a Newton step 8 and 1 more: from tau0 a node needs 8 to
// 10 sweeps and a warp 12 to 18, from the guess 3 (4096^2 cavity, n = 0.5, developed flow, us a step,
// plain sweeps / from the guess: FP32 Yu 278 / 201, Chai 288 / 209, 1024^2 FP64 2.8 / 1.0 ms; at rest, where two plain
// sweeps do, the guess costs 1%).
template <int CLOSURE, class RS>
__device__ __forceinline__ RS tau_fixed_point(RS qa, RS qb2, RS qc, const StepArgs<RS>& a) {
    RS tau = a.tau0;
    if constexpr (CLOSURE == CL_SMAG) {
        for (int it = 0; it < a.smag_iters; ++it) {
            const RS s = c_rcp(tau);
            const RS tn = fma(a.smag_c3, c_sqrt(RS(2) * fma(fma(qc, s, qb2), s, qa)), a.tau0);
            if (tn == tau) break;
            tau = tn;
        }
    } else {
        if (a.pl_nm1 == RS(0)) {  // n = 1: F does not depend on tau (1025x1023 11.3 us a step, by sweeps 12.9)
            RS tn = a.pl_k3 + RS(0.5);
            if (!(tn >= a.pl_tau_min)) tn = a.pl_tau_min;
            return tn > a.pl_tau_max ? a.pl_tau_max : tn;
        }
        const bool newton = a.pl_guess.on != 0;
        if (newton) tau = power_law_start(qc, a);
        for (int it = 1; it <= a.pl_max_iter; ++it) {
            const RS s = c_rcp(tau);
            const RS r = fma(fma(qc, s, qb2), s, qa);
            const RS t = fma(a.pl_k3, strain_pow(RS(2) * r, a.pl_nm1), RS(0.5));
            RS tn = t;
            if (!(tn >= a.pl_tau_min)) tn = a.pl_tau_min;
            if (tn > a.pl_tau_max) tn = a.pl_tau_max;
            const RS diff = tn - tau;
            tau = tn;
            if (r_abs(diff) <= a.pl_tol * tn) break;
            // Newton: dF/dtau = -e / r; not where it nears 1, and plain sweeps should eight steps not do
            if (newton && tn == t && it <= 8) {
                const RS e = (t - RS(0.5)) * a.pl_nm1 * (s * s) * fma(qc, s, RS(0.5) * qb2);
                const RS den = r + e;
                if (den > RS(0.25) * r) {
                    tau = fma(-diff * e, c_rcp(den), tn);  // tau + diff r / (r + e), from F(tau)
                    if (!(tau >= a.pl_tau_min)) tau = a.pl_tau_min;
                    if (tau > a.pl_tau_max) tau = a.pl_tau_max;
                }
            }
        }
    }
    return tau;
}

// L2 eviction priority for per-node fields that every step reads again while the populations
// stream past: the force field (read-only) and the lagged closure's stored tau (read and rewritten
// by its own node each step).  Their loads and stores carry an evict_last policy, so the field
// (12 or 4 B per node in FP32) stays in L2 across the steps of a launch instead of coming from HBM
// every step.  A hint only: the data are the same either way.  Measured on a GB300: one 25 MB
// field stays (the same loads without the policy run at the old speed); two such fields hinted
// at once in the adjoint's reverse step (force field and gradient accumulator) both kept
// streaming from HBM, so only the force field carries the hint there.
__device__ __forceinline__ unsigned long long l2_keep() {
    unsigned long long pol;
    asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
// read-only field (non-coherent path), evict_last in L2
template <class RS>
__device__ __forceinline__ RS ld_keep(const RS* p) {
    const unsigned long long pol = l2_keep();
    if constexpr (std::is_same<RS, double>::value) {
        double v;
        asm("ld.global.nc.L2::cache_hint.f64 %0, [%1], %2;" : "=d"(v) : "l"(p), "l"(pol));
        return v;
    } else {
        float v;
        asm("ld.global.nc.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(p), "l"(pol));
        return v;
    }
}
// an aligned FP32 pair (p 8-byte aligned) of a read-only field, evict_last in L2
__device__ __forceinline__ float2 ld2_keep(const float* p) {
    const unsigned long long pol = l2_keep();
    float2 v;
    asm("ld.global.nc.L2::cache_hint.v2.f32 {%0, %1}, [%2], %3;" : "=f"(v.x), "=f"(v.y) : "l"(p), "l"(pol));
    return v;
}
// a field value written by another block earlier in the launch: loaded through L2 (asm volatile,
// so its issue point stays where it is written) and stored back, both evict_last in L2
template <class RS>
__device__ __forceinline__ RS load_early_keep(const RS* p) {
    const unsigned long long pol = l2_keep();
    if constexpr (std::is_same<RS, double>::value) {
        double v;
        asm volatile("ld.global.cg.L2::cache_hint.f64 %0, [%1], %2;" : "=d"(v) : "l"(p), "l"(pol));
        return v;
    } else {
        float v;
        asm volatile("ld.global.cg.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(p), "l"(pol));
        return v;
    }
}
// the same load without the eviction policy
template <class RS>
__device__ __forceinline__ RS load_early(const RS* p) {
    if constexpr (std::is_same<RS, double>::value) {
        double v;
        asm volatile("ld.global.cg.f64 %0, [%1];" : "=d"(v) : "l"(p));
        return v;
    } else {
        float v;
        asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(v) : "l"(p));
        return v;
    }
}
template <class RS>
__device__ __forceinline__ void st_keep(RS* p, RS v) {
    const unsigned long long pol = l2_keep();
    if constexpr (std::is_same<RS, double>::value)
        asm volatile("st.global.L2::cache_hint.f64 [%0], %1, %2;" ::"l"(p), "d"(v), "l"(pol) : "memory");
    else
        asm volatile("st.global.L2::cache_hint.f32 [%0], %1, %2;" ::"l"(p), "f"(v), "l"(pol) : "memory");
}

// Deviatoric Smagorinsky, tau = tau0 + 3 Cs^2 |S_d(1/tau)|.  On these bases the rate-free part A is
// isotropic and B is traceless, so S_d = s B and tau is the larger root of
// tau^2 - tau0 tau - 3 Cs^2 |B| = 0, |B| = sqrt(2 B:B).
template <class RS>
__device__ __forceinline__ RS tau_deviatoric(RS qc, const StepArgs<RS>& a) {
    const RS b = c_sqrt(RS(2) * qc);
    return RS(0.5) * (a.tau0 + c_sqrt(fma(a.tau0, a.tau0, RS(4) * a.smag_c3 * b)));
}

// Returns tau, sets snu = 1/tau and S = A + snu B.  The lagged closure collides with tau_prev, the
// tau stored at `node` (loaded by the caller together with the populations), and in a step (not a
// read-out) stores tau0 + 3 Cs^2 |S| there for the next step.
template <class L, class R, int CLOSURE, bool STEP, class RS>
__device__ __forceinline__ R solve_tau(const R (&A)[L::NS], const R (&B)[L::NS], const StepArgs<RS>& a,
                                       R (&S)[L::NS], R& snu, int node, R tau_prev = R(0.0f)) {
    if constexpr (CLOSURE == CL_NEWTON) {
        snu = R(a.s[L::NU0]);
        affine<L>(A, B, snu, S);
        return R(a.tau0);
    } else if constexpr (CLOSURE == CL_SMAG_LAGGED) {
        const R tau = tau_prev;
        snu = c_rcp(tau);
        affine<L>(A, B, snu, S);
        if constexpr (STEP)
            st_keep(a.tau_field + node, RS(fma(a.smag_c3, c_sqrt(RS(2) * strain_dot<L>(S, S)), a.tau0)));
        return tau;
    } else if constexpr (CLOSURE == CL_SMAG_DEV) {
        const R tau = tau_deviatoric(strain_dot<L>(B, B), a);
        snu = c_rcp(tau);
        affine<L>(A, B, snu, S);
        return tau;
    } else {
        const R qa = strain_dot<L>(A, A), qb2 = R(2.0f) * strain_dot<L>(A, B), qc = strain_dot<L>(B, B);
        const R tau = tau_fixed_point<CLOSURE>(qa, qb2, qc, a);
        snu = c_rcp(tau);
        affine<L>(A, B, snu, S);
        return tau;
    }
}

// ------------------------------------------------------------------------------------------
// pull streaming

// Pre-collision populations of node (x,y,z).  Interior rows (y, z away from the faces, and x
// away from non-periodic x faces) read population i at node + (x wrap) - c_iy nx - c_iz nx ny,
// the last two terms being the same for the whole warp; nodes on a periodic boundary row or plane
// with no wall next to them read the same way with the y and z wraps applied by index (a separate
// branch, so the interior code stays as short); the rest take the general rule:
// periodic faces wrap, a population whose source lies behind a wall is reflected from the
// opposite population of the same node, plus the moving-wall term when it crosses exactly one
// moving face.
template <class L, class ST, class RS>
__device__ __forceinline__ bool interior_rows(const StepArgs<RS>& a, int xlo, int xhi, int y, int z) {
    const bool xwall = (a.wall_mask & 3) != 0;
    bool fast = y > 0 && y < a.ny - 1 && (!xwall || (xlo > 0 && xhi < a.nx - 1));
    if constexpr (L::D == 3) fast = fast && z > 0 && z < a.nz - 1;
    return fast;
}

// no wall face next to the node (its periodic faces wrap by index)
template <class L, class ST, class RS>
__device__ __forceinline__ bool no_wall_next(const StepArgs<RS>& a, int x, int y, int z) {
    const int w = a.wall_mask;  // bit f: face f (-x, +x, -y, +y, -z, +z) is a wall
    bool ok = !(w & 3) || (x > 0 && x < a.nx - 1);
    ok = ok && (!(w & 12) || (y > 0 && y < a.ny - 1));
    if constexpr (L::D == 3) ok = ok && (!(w & 48) || (z > 0 && z < a.nz - 1));
    return ok;
}

// neighbour offsets along y and z with the periodic wrap: the source of c = +1 is one step back
struct WrapYZ {
    int ym, yp, zm, zp;
    __device__ __forceinline__ WrapYZ(int y, int z, int nx, int ny, int nz) {
        const int nxy = nx * ny;
        ym = y == 0 ? (ny - 1) * nx : -nx;
        yp = y == ny - 1 ? -(ny - 1) * nx : nx;
        zm = z == 0 ? (nz - 1) * nxy : -nxy;
        zp = z == nz - 1 ? -(nz - 1) * nxy : nxy;
    }
    template <int cy, int cz>
    __device__ __forceinline__ int off() const {
        return (cy > 0 ? ym : (cy < 0 ? yp : 0)) + (cz > 0 ? zm : (cz < 0 ? zp : 0));
    }
};

// population load: COH selects the coherent (L2) path
template <bool COH, class ST>
__device__ __forceinline__ typename Store<ST>::R ldp(const ST* p) {
    if constexpr (COH)
        return Store<ST>::ldc(p);
    else
        return Store<ST>::ld(p);
}
template <bool COH, class ST>
__device__ __forceinline__ F2 ldp2(const ST* p) {
    if constexpr (COH)
        return Store<ST>::ld2c(p);
    else
        return Store<ST>::ld2(p);
}

template <class L, class ST, bool COH = false, class RS>
__device__ __forceinline__ void pull_general(const StepArgs<RS>& a, int x, int y, int z, RS (&f)[L::Q],
                                             long long es = 0) {
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const int node = (z * ny + y) * nx + x;
    const int dims[3] = {nx, ny, nz};
    const int pos[3] = {x, y, z};
    sfor<L::Q>([&](auto i) {
        int s[3];
        int nout = 0, face = -1;
        sfor<3>([&](auto ax) {
            constexpr int cax = L::c(CV(i), CV(ax));
            s[ax] = pos[ax] - cax;
            if constexpr (cax != 0) {
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
            f[i] = ldp<COH>(static_cast<const ST*>(a.srcp[CV(i)]) + es + ((s[2] * ny + s[1]) * nx + s[0]));
        } else {
            RS v = ldp<COH>(static_cast<const ST*>(a.srcp[opp<L>(CV(i))]) + es + node);
            if (nout == 1 && ((a.lid_mask >> face) & 1)) {
                const RS cu = RS(L::c(CV(i), 0)) * a.lid[face][0] + RS(L::c(CV(i), 1)) * a.lid[face][1] +
                              RS(L::c(CV(i), 2)) * a.lid[face][2];
                v += RS(double(6 * L::wnum(CV(i))) / L::WDEN) * a.rho0 * cu;  // 2 w_i rho0 (c.u)/cs^2 = 6 w_i rho0 c.u
            }
            f[i] = v;
        }
    });
}

template <class L, class ST, bool COH = false, class RS>
__device__ __forceinline__ void pull(const StepArgs<RS>& a, int x, int y, int z, RS (&f)[L::Q], long long es = 0) {
    const int nx = a.nx, nxy = a.nx * a.ny;
    const int node = z * nxy + y * nx + x;
    const int dxm = x == 0 ? nx - 1 : -1;      // source of c_x = +1: x - 1 (wrapped)
    const int dxp = x == nx - 1 ? 1 - nx : 1;  // source of c_x = -1: x + 1 (wrapped)
    if (interior_rows<L, ST>(a, x, x, y, z)) {
        sfor<L::Q>([&](auto i) {
            constexpr int cx = L::c(CV(i), 0), cy = L::c(CV(i), 1), cz = L::c(CV(i), 2);
            const int off = node + (cx > 0 ? dxm : (cx < 0 ? dxp : 0)) - (cy * nx + cz * nxy);
            f[i] = ldp<COH>(static_cast<const ST*>(a.srcp[CV(i)]) + es + off);
        });
        return;
    }
    if (no_wall_next<L, ST>(a, x, y, z)) {  // on a periodic boundary row or plane: wrap y and z too
        const WrapYZ w(y, z, nx, a.ny, a.nz);
        sfor<L::Q>([&](auto i) {
            constexpr int cx = L::c(CV(i), 0), cy = L::c(CV(i), 1), cz = L::c(CV(i), 2);
            const int off = node + (cx > 0 ? dxm : (cx < 0 ? dxp : 0)) + w.template off<cy, cz>();
            f[i] = ldp<COH>(static_cast<const ST*>(a.srcp[CV(i)]) + es + off);
        });
        return;
    }
    pull_general<L, ST, COH>(a, x, y, z, f, es);
}

// Two nodes (x0, x0 + 1), x0 even, nx even: populations with c_x = 0 come as one aligned pair,
// the others as two scalar loads (x wrap applied per node); periodic boundary rows and planes
// with no wall next to either node wrap y and z by index, as in the one-node pull.
template <class L, class ST, bool COH = false>
__device__ __forceinline__ void pull2(const StepArgs<float>& a, int x0, int y, int z, F2 (&f)[L::Q]) {
    const int nx = a.nx, nxy = a.nx * a.ny;
    const int node = z * nxy + y * nx + x0;
    if (interior_rows<L, ST>(a, x0, x0 + 1, y, z)) {
        const int dxm = x0 == 0 ? nx - 1 : -1;          // node 0, c_x = +1: x0 - 1 (wrapped)
        const int dxp = x0 + 2 == nx ? 2 - nx : 2;      // node 1, c_x = -1: x0 + 2 (wrapped)
        sfor<L::Q>([&](auto i) {
            constexpr int cx = L::c(CV(i), 0), cy = L::c(CV(i), 1), cz = L::c(CV(i), 2);
            const ST* p = static_cast<const ST*>(a.srcp[CV(i)]) + (node - (cy * nx + cz * nxy));
            if constexpr (cx == 0)
                f[i] = ldp2<COH>(p);
            else if constexpr (cx > 0)
                f[i] = F2(ldp<COH>(p + dxm), ldp<COH>(p));
            else
                f[i] = F2(ldp<COH>(p + 1), ldp<COH>(p + dxp));
        });
        return;
    }
    if (no_wall_next<L, ST>(a, x0, y, z) && no_wall_next<L, ST>(a, x0 + 1, y, z)) {
        // on a periodic boundary row or plane: the same loads with the y and z wraps by index
        const WrapYZ w(y, z, nx, a.ny, a.nz);
        const int dxm = x0 == 0 ? nx - 1 : -1;
        const int dxp = x0 + 2 == nx ? 2 - nx : 2;
        sfor<L::Q>([&](auto i) {
            constexpr int cx = L::c(CV(i), 0), cy = L::c(CV(i), 1), cz = L::c(CV(i), 2);
            const ST* p = static_cast<const ST*>(a.srcp[CV(i)]) + (node + w.template off<cy, cz>());
            if constexpr (cx == 0)
                f[i] = ldp2<COH>(p);
            else if constexpr (cx > 0)
                f[i] = F2(ldp<COH>(p + dxm), ldp<COH>(p));
            else
                f[i] = F2(ldp<COH>(p + 1), ldp<COH>(p + dxp));
        });
        return;
    }
    float f0[L::Q], f1[L::Q];
    pull_general<L, ST, COH>(a, x0, y, z, f0);
    pull_general<L, ST, COH>(a, x0 + 1, y, z, f1);
    sfor<L::Q>([&](auto i) { f[i] = F2(f0[i], f1[i]); });
}

// ------------------------------------------------------------------------------------------
// the fused step

// Programmatic dependent launch.  A step launched with the programmatic-serialization attribute
// may become resident while the previous kernel of the stream is finishing; griddepcontrol.wait
// returns once that kernel has completed and its memory operations are visible, so it precedes
// every load.  launch_dependents lets the next such step be scheduled as soon as every block of
// this one has issued it; issued at block start, that happens once the last blocks are resident,
// so waiting blocks of the next step only take slots freed by this one.  Launched without the
// attribute, both instructions have no effect.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// opposite-pair sums and differences of the pulled populations
template <class L, class R>
__device__ __forceinline__ void pair_sums(const R (&f)[L::Q], R (&P)[L::NP], R (&Dd)[L::NP]) {
    sfor<L::NP>([&](auto p) {
        P[p] = f[L::pa(CV(p))] + f[L::pb(CV(p))];
        Dd[p] = f[L::pa(CV(p))] - f[L::pb(CV(p))];
    });
}

// the node's force density: its entry of the force field, or the uniform force
template <class L, bool FORCE, class RS, class R>
__device__ __forceinline__ void node_force(const StepArgs<RS>& a, int node, R (&F)[3]) {
    sfor<3>([&](auto d) { F[d] = R(0.0f); });
    if constexpr (FORCE) {
        if (a.force_field) {
            const long long N = (long long)a.nx * a.ny * a.nz;  // component offsets exceed 2^31 on big grids
            sfor<L::D>([&](auto d) { F[d] = ld_keep(a.force_field + CV(d) * N + node); });
        } else {
            sfor<L::D>([&](auto d) { F[d] = R(a.F[d]); });
        }
    }
}

// delta rho, j = sum c f + F/2 and u = j / rho0; on the Yu route with all moments m = T f
template <class L, int FORMULA, bool FORCE, class R>
__device__ __forceinline__ void conserved_moments(R f0, const R (&P)[L::NP], const R (&Dd)[L::NP], const R (&F)[3],
                                                  R ir0, R& drho, R (&j)[3], R (&u)[3], R (&m)[L::Q]) {
    j[2] = u[2] = R(0.0f);
    if constexpr (FORMULA == F_YU) {
        Xf<L>::forward(f0, P, Dd, m);
        drho = m[0];
        j[0] = FORCE ? fma(R(0.5f), F[0], m[3]) : m[3];
        j[1] = FORCE ? fma(R(0.5f), F[1], m[5]) : m[5];
        if constexpr (L::D == 3) j[2] = FORCE ? fma(R(0.5f), F[2], m[7]) : m[7];
    } else {
        drho = f0;
        sfor<L::NP>([&](auto p) { drho += P[p]; });
        sfor<L::D>([&](auto d) {
            R acc = nzero<R>();
            sfor<L::NP>([&](auto p) { acc = cadd<L::c(L::pa(CV(p)), CV(d))>(acc, Dd[p]); });
            j[d] = FORCE ? fma(R(0.5f), F[d], acc) : acc;
        });
    }
    sfor<L::D>([&](auto d) { u[d] = j[d] * ir0; });
}

// non-equilibrium moments mn = T (f - f_eq + Fbar/2) of the non-conserved rows, with TF = T Fbar.  Yu
// route: the moments of f less the closed-form equilibrium moments.  Chai route: the moments of the
// non-equilibrium distributions (in opposite-pair form).
template <class L, int FORMULA, bool FORCE, class R>
__device__ __forceinline__ void noneq_moments(R f0, const R (&P)[L::NP], const R (&Dd)[L::NP], const R (&F)[3],
                                              R drho, const R (&j)[3], const R (&u)[3], const R (&m)[L::Q],
                                              R (&mn)[L::Q], R (&TF)[L::Q]) {
    if constexpr (FORCE) Eq<L>::tforce(u, F, TF);
    if constexpr (FORMULA == F_YU) {
        R meq[L::Q];
        Eq<L>::meq(drho, j, u, meq);
        sfor<L::Q>([&](auto k) {
            if constexpr (L::conserved(CV(k)))
                mn[k] = R(0.0f);
            else if constexpr (Eq<L>::ghost(CV(k)))
                mn[k] = m[k];
            else if constexpr (FORCE)
                mn[k] = fma(R(0.5f), TF[k], m[k] - meq[k]);
            else
                mn[k] = m[k] - meq[k];
        });
    } else {
        R fn0, Pn[L::NP], Dn[L::NP];
        noneq_pairs<L, FORCE>(f0, P, Dd, drho, j, u, F, fn0, Pn, Dn);
        Xf<L>::forward(fn0, Pn, Dn, mn);
    }
}

// Chai's formula with fixed rates takes each viscous rate as given, so S does not split
template <int CLOSURE, int FORMULA>
constexpr bool rates_known() {
    return CLOSURE == CL_NEWTON && FORMULA == F_CHAI;
}

// S = A + s_nu B by the route's formula (B = 0 with the rates known)
template <class L, int CLOSURE, int FORMULA, class RS, class R>
__device__ __forceinline__ void strain_split(const StepArgs<RS>& a, const R (&mn)[L::Q], R ir0, R (&A)[L::NS],
                                             R (&B)[L::NS]) {
    if constexpr (FORMULA == F_YU) {
        Eq<L>::yu_split(mn, R(a.s[1] * RS(Eq<L>::YU_A)) * ir0, ir0, A, B);
    } else {
        constexpr bool KNOWN = rates_known<CLOSURE, FORMULA>();
        const R kS = R(-1.5f) * ir0;  // -1 / (2 rho0 cs^2)
        R Dn[L::Q];
        sfor<L::Q>([&](auto k) {
            if constexpr (L::viscous(CV(k)) && !KNOWN)
                Dn[k] = cst<R>(1.0 / norm2<L>(CV(k))) * mn[k];
            else if constexpr (!L::conserved(CV(k)))
                Dn[k] = R(a.skn[k]) * mn[k];
        });
        chai_contract<L>(Dn, kS, [](int k) { return !L::conserved(k) && (KNOWN || !L::viscous(k)); }, A);
        if constexpr (KNOWN)
            sfor<L::NS>([&](auto c) { B[c] = R(0.0f); });
        else
            chai_contract<L>(Dn, kS, [](int k) { return L::viscous(k); }, B);
    }
}

// Everything of a step after the pull, for the node `node`: moments, strain rate by the chosen route,
// closure, relaxation, force; sink(i, v) takes f*_i.  With fixed rates a step needs no S and relaxes each viscous
// moment at its own rate.
template <class L, class ST, int CLOSURE, int FORMULA, bool FORCE, class Sink>
__device__ __forceinline__ void collide(const StepArgs<typename Store<ST>::R>& a, typename Store<ST>::R (&f)[L::Q],
                                        int node, Sink&& sink) {
    using R = typename Store<ST>::R;
    constexpr int Q = L::Q, NS = L::NS, NP = L::NP;

    R P[NP], Dd[NP], F[3];
    pair_sums<L>(f, P, Dd);
    node_force<L, FORCE>(a, node, F);
    // the lagged closure's stored tau, loaded next to the populations so its latency overlaps theirs
    // (an asm volatile load keeps it there instead of next to its use after the moment arithmetic)
    R tau_prev = R(0.0f);
    if constexpr (CLOSURE == CL_SMAG_LAGGED) tau_prev = load_early_keep(a.tau_field + node);
    const R ir0 = R(a.inv_rho0);
    R drho, j[3], u[3], m[Q], mn[Q], TF[Q];
    conserved_moments<L, FORMULA, FORCE>(f[0], P, Dd, F, ir0, drho, j, u, m);
    noneq_moments<L, FORMULA, FORCE>(f[0], P, Dd, F, drho, j, u, m, mn, TF);
    // every collision increment D_k = (s_k mn_k - TF_k) / |T_k|^2 that does not involve an unknown
    // viscous rate is finished before the closure, so only the viscous moments (and their force terms)
    // stay live across the fixed point
    constexpr bool KNOWN = CLOSURE == CL_NEWTON;  // every rate given: S is not needed
    R Dk[Q], tv[Q];
    sfor<Q>([&](auto k) {
        constexpr double inv_n = 1.0 / norm2<L>(CV(k));
        constexpr bool has_tf = FORCE && !Eq<L>::ghost(CV(k));
        if constexpr (L::conserved(CV(k))) {
            if constexpr (FORCE)
                Dk[k] = cst<R>(-inv_n) * TF[k];
            else
                Dk[k] = R(0.0f);
        } else {
            if constexpr (has_tf) tv[k] = cst<R>(-inv_n) * TF[k];
            if constexpr (!L::viscous(CV(k)) || KNOWN) {
                if constexpr (has_tf)
                    Dk[k] = fma(R(a.skn[k]), mn[k], tv[k]);
                else
                    Dk[k] = R(a.skn[k]) * mn[k];
            }
        }
    });
    if constexpr (!KNOWN) {
        R A[NS], B[NS], S[NS], snu;
        strain_split<L, CLOSURE, FORMULA>(a, mn, ir0, A, B);
        solve_tau<L, R, CLOSURE, true>(A, B, a, S, snu, node, tau_prev);
        sfor<Q>([&](auto k) {
            if constexpr (L::viscous(CV(k))) {
                constexpr double inv_n = 1.0 / norm2<L>(CV(k));
                if constexpr (FORCE)
                    Dk[k] = fma(snu * cst<R>(inv_n), mn[k], tv[k]);
                else
                    Dk[k] = (snu * cst<R>(inv_n)) * mn[k];
            }
        });
    }
    // f*_i = f_i - out_i; with a force, the conserved moments 3, 5, 7 (D2Q9: 3, 5) carry -TF_k; TF_0 = 0
    R out[Q];
    Xf<L>::template backward<FORCE ? mask_all_but_density<L>() : mask_nonconserved<L>()>(Dk, out);
    sfor<Q>([&](auto i) { sink(i, f[i] - out[i]); });
}

// The Guo-type discrete force in opposite-pair form (noneq_pairs): even parts E, c.F of each pair (odd part 3 w c.F)
// and u.F (rest -3 w0 u.F)
template <class L, class R>
__device__ __forceinline__ void force_pairs(const R (&u)[3], const R (&F)[3], R& uF, R (&E)[L::NP], R (&cF)[L::NP]) {
    uF = fma(u[0], F[0], fma(u[1], F[1], u[2] * F[2]));
    sfor<L::NP>([&](auto p) {
        constexpr int i = L::pa(CV(p));
        constexpr int cx = L::c(i, 0), cy = L::c(i, 1), cz = L::c(i, 2);
        constexpr double w = double(L::wnum(i)) / L::WDEN;
        const R cu = cadd<cz>(cadd<cy>(cadd<cx>(nzero<R>(), u[0]), u[1]), u[2]);
        cF[p] = cadd<cz>(cadd<cy>(cadd<cx>(nzero<R>(), F[0]), F[1]), F[2]);
        E[p] = fma(cst<R>(9.0 * w) * cu, cF[p], cst<R>(-3.0 * w) * uF);
    });
}

// Chai's route of a 16-bit lattice at one node (nx odd; step_pair.cuh has the pair): as collide, with Omega formed
// in the q directions (omega_split), f* = f - Omega + Fbar.
template <class L, class ST, int CLOSURE, bool FORCE, class Sink>
__device__ __forceinline__ void collide_omega(const StepArgs<typename Store<ST>::R>& a,
                                              typename Store<ST>::R (&f)[L::Q], int node, Sink&& sink) {
    using R = typename Store<ST>::R;
    constexpr int Q = L::Q, NS = L::NS, NP = L::NP;
    R P[NP], Dd[NP], F[3];
    pair_sums<L>(f, P, Dd);
    node_force<L, FORCE>(a, node, F);
    const R ir0 = R(a.inv_rho0);
    R drho, j[3], u[3], m[Q], mn[Q], fn0, Pn[NP], Dn[NP];
    conserved_moments<L, F_CHAI, FORCE>(f[0], P, Dd, F, ir0, drho, j, u, m);
    noneq_pairs<L, FORCE>(f[0], P, Dd, drho, j, u, F, fn0, Pn, Dn);
    Xf<L>::forward(fn0, Pn, Dn, mn);
    constexpr double w0 = double(L::wnum(0)) / L::WDEN;
    R uF, FE[NP], cF[NP];
    if constexpr (FORCE) force_pairs<L>(u, F, uF, FE, cF);
    R Ef0, Ef[NP], Of[NP], Ev[NP], A[NS], B[NS], S[NS], snu;
    omega_split<L>(a, mn, ir0, Ef0, Ef, Of, Ev, A, B);
    // everything but s_nu Omega_v is folded into f now, so that only f and Omega_v stay live across the closure
    f[0] -= Ef0;
    if constexpr (FORCE) f[0] = fma(cst<R>(-3.0 * w0), uF, f[0]);
    sfor<NP>([&](auto p) {
        R e = Ef[p], o = Of[p];
        if constexpr (FORCE) {
            constexpr double w = double(L::wnum(L::pa(CV(p)))) / L::WDEN;
            e -= FE[p];
            o = fma(cst<R>(-3.0 * w), cF[p], o);
        }
        f[L::pa(CV(p))] -= e + o;
        f[L::pb(CV(p))] -= e - o;
    });
    solve_tau<L, R, CLOSURE, true>(A, B, a, S, snu, node);
    sink(std::integral_constant<int, 0>{}, f[0]);
    sfor<NP>([&](auto p) {
        const R e = snu * Ev[p];
        sink(std::integral_constant<int, L::pa(CV(p))>{}, f[L::pa(CV(p))] - e);
        sink(std::integral_constant<int, L::pb(CV(p))>{}, f[L::pb(CV(p))] - e);
    });
}

// The collision with f* stored at the node.  ds shifts the populations' destination by that many elements (a
// launch that writes each step to its own buffer of a ring); the pull's es does the same for the source.
template <class L, class ST, int CLOSURE, int FORMULA, bool FORCE>
__device__ __forceinline__ void step_body(const StepArgs<typename Store<ST>::R>& a, typename Store<ST>::R (&f)[L::Q],
                                          int node, long long ds = 0) {
    auto sink = [&](auto i, auto v) { Store<ST>::st(static_cast<ST*>(a.dstp[CV(i)]) + ds + node, v); };
    if constexpr (sizeof(ST) == 2 && FORMULA == F_CHAI && CLOSURE != CL_NEWTON)
        collide_omega<L, ST, CLOSURE, FORCE>(a, f, node, sink);
    else
        collide<L, ST, CLOSURE, FORMULA, FORCE>(a, f, node, sink);
}

// Which node(s) a thread takes: PER x-adjacent nodes each (nx a multiple of PER), in node order over the
// computed planes, so that rows of any length fill the blocks (GLUPS, blocks cut at the row ends / node order: FP32
// 200x150x97 channel 35.8 / 40.6, 97x150x97 28.6 / 37.1, 80^3 box 37.1 / 45.9, 301x301x199 39.0 / 45.3, FP16
// 200x150x97 42.8 / 50.9, 96^3 48.1 / 63.8; but see whole_rows).  Where rows fill whole blocks
// anyway (nx.m = 0) the grid gives x, y and z directly, without the two divisions; the FP32 and FP64 steps
// are built for each map, since choosing at run time cost them up to 8% (121x89x38 channel).
struct NodeMap {
    FastDiv nx, ny;  // thread positions per row, rows per plane
    int threads;     // thread positions in all
};
template <int PER, class RS>
inline NodeMap node_map(const StepArgs<RS>& a) {
    return {fast_div((unsigned)(a.nx / PER)), fast_div((unsigned)a.ny), a.nx / PER * a.ny * a.nzc};
}
template <int PER, class RS>
__device__ __forceinline__ bool node_in_grid(const StepArgs<RS>& a, int& x, int& y, int& z) {
    x = PER * (blockIdx.x * blockDim.x + threadIdx.x);
    y = blockIdx.y * blockDim.y + threadIdx.y;
    z = blockIdx.z + a.z0;
    return x < a.nx && y < a.ny;
}
template <int PER, class RS>
__device__ __forceinline__ bool node_in_order(const StepArgs<RS>& a, const NodeMap& g, int& x, int& y, int& z) {
    const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (unsigned)g.threads) return false;
    const int row = div_fast((int)t, g.nx), zz = div_fast(row, g.ny);
    x = PER * (int)t - row * a.nx;
    y = row - zz * a.ny;
    z = zz + a.z0;
    return true;
}
template <int PER, class RS>
__device__ __forceinline__ bool node_at(const StepArgs<RS>& a, const NodeMap& g, int& x, int& y, int& z) {
    return g.nx.m == 0 ? node_in_grid<PER>(a, x, y, z) : node_in_order<PER>(a, g, x, y, z);
}
// the launch geometry of a map for blocks of `threads`; rows that waste at most 1/waste of themselves in
// idle threads (0: none) count as filling their blocks
template <int PER, class RS>
inline NodeMap node_grid(const StepArgs<RS>& a, int threads, int waste, dim3* grid) {
    NodeMap g = node_map<PER>(a);
    const int row = a.nx / PER, blocks = (row + threads - 1) / threads;
    if ((long long)blocks * threads - row <= (waste ? row / waste : 0)) {
        g.nx.m = 0;
        *grid = dim3(blocks, a.ny, a.nzc);
    } else {
        *grid = dim3((unsigned)((g.threads + (long long)threads - 1) / threads));
    }
    return g;
}

// One node per thread.  The bound names no minimum of resident blocks for the 16-bit and FP32 3D lattices: a
// minimum of one changes ptxas's register allocation (more registers, fewer resident blocks).  FP64 names one
// that leaves it more registers than it takes unasked (up to 128 in 3D, 64 in 2D): bound by the FP64 pipe, the step
// gains by holding values instead of forming them again (us a step, unasked / bounded: D3Q19 256x128x128 channel Yu
// 3250 at 106 registers / 2918 at 116, 128x128x64 Newtonian box Chai 495 / 451, D3Q15 256x128x64 channel Yu 1355 / 1276,
// 1000^2 D2Q9 Newtonian Chai 205 / 186; a cap of 80 registers in 3D was the slowest).  FP32 D2Q9 is
// held to 16 blocks (32 registers, full occupancy; the power law spills up to 12 values there): 4096^2
// power-law cavity, developed n = 0.5 flow, Yu / Chai 83 / 79 GLUPS, at 12 blocks 80 / 77, at 10 71 / 68.
template <class L, class ST>
constexpr int step_min_blocks() {
    if (sizeof(ST) == 8) return L::Q == 9 ? 8 : 4;
    return L::Q == 9 && sizeof(ST) == 4 ? 16 : 0;
}

template <class L, class ST, int CLOSURE, int FORMULA, bool FORCE, bool GRID>
__global__ void __launch_bounds__(128, step_min_blocks<L, ST>())
    k_step(const StepArgs<typename Store<ST>::R> a, const NodeMap g) {
    pdl_wait();     // the previous step's stores are complete and visible from here on
    // Every block has started: the next step may be scheduled into freed slots.  Not in FP64, whose blocks wait
    // for their SM's share of the FP64 pipe: blocks of the next step that come early leave the rest to
    // whichever SM is done first, and the SMs end up with unequal shares (40^3 1.85 against 2.39 GLUPS,
    // 119x891 D2Q9 2.90 against 4.15).
    if constexpr (sizeof(ST) != 8) pdl_release();
    int x, y, z;
    if (!(GRID ? node_in_grid<1>(a, x, y, z) : node_in_order<1>(a, g, x, y, z))) return;
    typename Store<ST>::R f[L::Q];
    pull<L, ST>(a, x, y, z, f);
    step_body<L, ST, CLOSURE, FORMULA, FORCE>(a, f, (z * a.ny + y) * a.nx + x);
}

}  // namespace lbm
