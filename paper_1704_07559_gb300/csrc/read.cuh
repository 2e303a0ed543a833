// read.cuh -- the read-outs of the state that the next step sees: S and tau, the macroscopic fields, and
// the global sums.
//
// Each pulls the populations as a step does and keeps only what it returns: the strain kernel the six
// moments of S and the closure, the macroscopic kernel the four conserved moments and no closure.  All are
// bound by reading the q populations (FP64 S by its FP64 operations).  As a run-time branch inside the step
// kernel they carried the step's registers and finished its collision increments first: on a
// 200x150x97 FP32 channel S by Chai's formula with tau took 80 us and the fields 81 us, here 50 and
// 39 (their bytes take 45 and 39 us at the measured copy bandwidth).
#pragma once

#include "launch.h"
#include "step.cuh"

namespace lbm {

template <class L, class ST, int CLOSURE, int FORMULA, bool FORCE>
__global__ void __launch_bounds__(128) k_strain(const StepArgs<typename Store<ST>::R> a, const NodeMap g) {
    using R = typename Store<ST>::R;
    pdl_wait();
    pdl_release();
    int x, y, z;
    if (!node_in_order<1>(a, g, x, y, z)) return;
    const int node = (z * a.ny + y) * a.nx + x;
    const long long N = (long long)a.nx * a.ny * a.nz;  // component offsets c*N exceed 2^31 on big grids
    R f[L::Q], P[L::NP], Dd[L::NP], F[3];
    pull<L, ST>(a, x, y, z, f);
    node_force<L, FORCE>(a, node, F);
    R tau_prev = R(0.0f);
    if constexpr (CLOSURE == CL_SMAG_LAGGED) tau_prev = load_early_keep(a.tau_field + node);
    pair_sums<L>(f, P, Dd);
    const R ir0 = R(a.inv_rho0);
    R drho, j[3], u[3], m[L::Q], mn[L::Q], TF[L::Q], A[L::NS], B[L::NS], S[L::NS], snu;
    conserved_moments<L, FORMULA, FORCE>(f[0], P, Dd, F, ir0, drho, j, u, m);
    noneq_moments<L, FORMULA, FORCE>(f[0], P, Dd, F, drho, j, u, m, mn, TF);
    strain_split<L, CLOSURE, FORMULA>(a, mn, ir0, A, B);
    const R tau = solve_tau<L, R, CLOSURE, false>(A, B, a, S, snu, node, tau_prev);
    sfor<L::NS>([&](auto c) { __stcs(a.S_out + CV(c) * N + node, S[c]); });
    if (a.tau_out) __stcs(a.tau_out + node, tau);
}

template <class L, class ST, int FORMULA, bool FORCE>
__global__ void __launch_bounds__(128) k_macro(const StepArgs<typename Store<ST>::R> a, const NodeMap g) {
    using R = typename Store<ST>::R;
    pdl_wait();
    pdl_release();
    int x, y, z;
    if (!node_in_order<1>(a, g, x, y, z)) return;
    const int node = (z * a.ny + y) * a.nx + x;
    const long long N = (long long)a.nx * a.ny * a.nz;
    R f[L::Q], P[L::NP], Dd[L::NP], F[3];
    pull<L, ST>(a, x, y, z, f);
    node_force<L, FORCE>(a, node, F);
    pair_sums<L>(f, P, Dd);
    R drho, j[3], u[3], m[L::Q];
    conserved_moments<L, FORMULA, FORCE>(f[0], P, Dd, F, R(a.inv_rho0), drho, j, u, m);
    if (a.drho_out) __stcs(a.drho_out + node, drho);
    if (a.u_out) sfor<L::D>([&](auto d) { __stcs(a.u_out + CV(d) * N + node, u[d]); });
}

// ------------------------------------------------------------------------------------------
// global sums: each block walks whole rows (fixed assignment, so the result is reproducible);
// each node's totals are formed in the compute type, then FP32 states accumulate them across nodes
// with an error-free two-sum (hi, lo) pair per component, FP64 states in plain FP64; per-block
// partials go to scratch as FP64 and one ordered pass adds them.  A thread waits for one node's
// populations at a time, so with FP32 arithmetic it fetches its next node's before adding the first's
// (the order of the additions is the same): 200x150x97 FP32 channel 57 us against 72 (its bytes: 33 us), and with
// every block resident (80 registers left the fourth of each SM to a second round) the three read-outs of a pass
// 178 us against 199.

constexpr int SUM_THREADS = 256;

template <class R>
struct Comp {
    R hi = R(0), lo = R(0);
    __device__ __forceinline__ void add(R x) {
        if constexpr (sizeof(R) == 4) {
            const R t = hi + x;
            const R bp = t - hi;
            lo += (hi - (t - bp)) + (x - bp);
            hi = t;
        } else {
            hi += x;
        }
    }
    __device__ __forceinline__ double value() const { return double(hi) + double(lo); }
};

// one node: its own totals in plain arithmetic, then one compensated add per component
template <class L, class R>
__device__ __forceinline__ void sum_node(const StepArgs<R>& a, const R (&f)[L::Q], int n, Comp<R> (&acc)[1 + L::D]) {
    const long long N = (long long)a.nx * a.ny * a.nz;  // component offsets c*N exceed 2^31 on big grids
    R m0 = nzero<R>(), mj[3] = {nzero<R>(), nzero<R>(), nzero<R>()};
    sfor<L::Q>([&](auto i) {
        m0 += f[i];
        sfor<L::D>([&](auto d) { mj[d] = cadd<L::c(CV(i), CV(d))>(mj[d], f[i]); });
    });
    acc[0].add(m0);
#pragma unroll
    for (int d = 0; d < L::D; ++d)
        acc[1 + d].add(fma(R(0.5), a.force_field ? a.force_field[d * N + n] : a.F[d], mj[d]));
}

// FP32 is held to 64 registers, so that the grid's four blocks per SM are resident together.
template <class L, class ST>
__global__ void __launch_bounds__(SUM_THREADS, sizeof(typename Store<ST>::R) == 4 ? SUM_PER_SM : 0)
    k_sums(const StepArgs<typename Store<ST>::R> a, double* __restrict__ partial) {
    using R = typename Store<ST>::R;
    constexpr int D = L::D;
    constexpr bool AHEAD = sizeof(R) == 4;
    const int rows = a.ny * a.nzc;  // the computed planes only (a halo plane belongs to a neighbour)
    Comp<R> acc[1 + D];
    int r = blockIdx.x, x = threadIdx.x;
    if (x >= a.nx) r = rows;
    // the thread's nodes in order: x, x + blockDim.x, ... of rows blockIdx.x, blockIdx.x + gridDim.x, ...
    auto fetch = [&](R (&f)[L::Q]) {
        const int z = r / a.ny + a.z0, y = r - (z - a.z0) * a.ny;
        pull<L, ST>(a, x, y, z, f);
        const int n = (z * a.ny + y) * a.nx + x;
        x += blockDim.x;
        if (x >= a.nx) {
            x = threadIdx.x;
            r += gridDim.x;
        }
        return n;
    };
    while (r < rows) {
        R f[L::Q];
        const int n = fetch(f);
        if (AHEAD && r < rows) {
            R g[L::Q];
            const int m = fetch(g);
            sum_node<L>(a, f, n, acc);
            sum_node<L>(a, g, m, acc);
        } else {
            sum_node<L>(a, f, n, acc);
        }
    }
    __shared__ double red[SUM_THREADS / 32][1 + D];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int c = 0; c <= D; ++c) {
        double v = acc[c].value();
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) red[warp][c] = v;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int c = 0; c <= D; ++c) {
            double v = 0.0;
            for (int w = 0; w < SUM_THREADS / 32; ++w) v += red[w][c];
            partial[blockIdx.x * (1 + D) + c] = v;
        }
    }
}

// Sums nblocks partial rows of `width` (at most 4) columns in a fixed order into out[0 .. width - 1]: thread t
// of 256 adds rows t, t + 256, ... of every column, then a tree over the threads.  With `flag`,
// out[width] = *flag (the multi-step launch's error word, read back with the sums in one copy).
__global__ void k_sums_final(const double* __restrict__ partial, int nblocks, int width, const int* flag,
                             double* __restrict__ out);

// ------------------------------------------------------------------------------------------
// launches

template <class L, class ST, int C, int F>
cudaError_t launch_strain_cf(const StepArgs<typename Store<ST>::R>& a, int force, cudaStream_t s) {
    // FP64: blocks of 64, as the step
    constexpr int T = sizeof(ST) == 8 ? 64 : 128;
    const NodeMap g = node_map<1>(a);
    const dim3 grid((unsigned)((g.threads + (long long)T - 1) / T));
    return force ? launch_pdl(k_strain<L, ST, C, F, true>, grid, dim3(T), s, a, g)
                 : launch_pdl(k_strain<L, ST, C, F, false>, grid, dim3(T), s, a, g);
}

template <class L, class ST, int C>
cudaError_t launch_strain_c(const StepArgs<typename Store<ST>::R>& a, int formula, int force, cudaStream_t s) {
    return formula == F_YU ? launch_strain_cf<L, ST, C, F_YU>(a, force, s) : launch_strain_cf<L, ST, C, F_CHAI>(a, force, s);
}

// EXTRA_CLOSURES as for the step
template <class L, class ST, bool EXTRA_CLOSURES>
cudaError_t launch_strain(const StepArgs<typename Store<ST>::R>& a, int closure, int formula, int force,
                          cudaStream_t s) {
    if (closure == CL_NEWTON) return launch_strain_c<L, ST, CL_NEWTON>(a, formula, force, s);
    if (closure == CL_SMAG) return launch_strain_c<L, ST, CL_SMAG>(a, formula, force, s);
    if constexpr (EXTRA_CLOSURES) {
        if (closure == CL_POWERLAW) return launch_strain_c<L, ST, CL_POWERLAW>(a, formula, force, s);
        if (closure == CL_SMAG_LAGGED) return launch_strain_c<L, ST, CL_SMAG_LAGGED>(a, formula, force, s);
        if (closure == CL_SMAG_DEV) return launch_strain_c<L, ST, CL_SMAG_DEV>(a, formula, force, s);
    }
    return cudaErrorNotSupported;
}

template <class L, class ST>
cudaError_t launch_macro(const StepArgs<typename Store<ST>::R>& a, int formula, int force, cudaStream_t s) {
    constexpr int T = sizeof(ST) == 8 ? 64 : 128;
    const NodeMap g = node_map<1>(a);
    const dim3 grid((unsigned)((g.threads + (long long)T - 1) / T));
    if (formula == F_YU)
        return force ? launch_pdl(k_macro<L, ST, F_YU, true>, grid, dim3(T), s, a, g)
                     : launch_pdl(k_macro<L, ST, F_YU, false>, grid, dim3(T), s, a, g);
    return force ? launch_pdl(k_macro<L, ST, F_CHAI, true>, grid, dim3(T), s, a, g)
                 : launch_pdl(k_macro<L, ST, F_CHAI, false>, grid, dim3(T), s, a, g);
}

template <class L, class ST>
cudaError_t launch_sums(const StepArgs<typename Store<ST>::R>& a, double* partial, int blocks, const int* flag,
                        double* out, cudaStream_t s) {
    k_sums<L, ST><<<blocks, SUM_THREADS, 0, s>>>(a, partial);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_sums_final<<<1, 256, 0, s>>>(partial, blocks, 1 + L::D, flag, out);
    return cudaGetLastError();
}

}  // namespace lbm

#define LBM_DEFINE_READ_ENTRY(TAG, L, ST, EXTRA_CLOSURES)                                                    \
    namespace lbm {                                                                                          \
    cudaError_t strain_##TAG(const StepArgs<Store<ST>::R>& a, int closure, int formula, int force,           \
                             cudaStream_t s) {                                                               \
        return launch_strain<L, ST, EXTRA_CLOSURES>(a, closure, formula, force, s);                          \
    }                                                                                                        \
    cudaError_t macro_##TAG(const StepArgs<Store<ST>::R>& a, int formula, int force, cudaStream_t s) {       \
        return launch_macro<L, ST>(a, formula, force, s);                                                    \
    }                                                                                                        \
    cudaError_t sums_##TAG(const StepArgs<Store<ST>::R>& a, double* partial, int blocks, const int* flag,    \
                           double* out, cudaStream_t s) {                                                    \
        return launch_sums<L, ST>(a, partial, blocks, flag, out, s);                                         \
    }                                                                                                        \
    }
