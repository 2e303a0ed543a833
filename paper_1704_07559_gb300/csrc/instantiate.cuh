// instantiate.cuh -- defines the step and init entry points of launch.h for one (lattice, storage)
// pair.  Included by one small translation unit per pair so the kernels compile in parallel.
#pragma once

#include "init.cuh"
#include "launch.h"
#include "step.cuh"
#include "step_pair.cuh"

namespace lbm {

// Between walls in y or z whole rows take the general pull, and in node order a warp across such a row and the next
// takes both branches.  Small lattices, whose slowest warps are their time, step there by blocks of whole rows
// (lattice_grid) while the lanes idle at row ends are under `idle`, one wave of blocks or, in FP32, half of one; FP64
// never, whose pipe bounds it.  us a step, whole rows / node order, channels, D3Q15: FP16 Newtonian 112x49x33 10.4 / 13.3, 60x90x90
// 19.3 / 23.2, 200x45x69 25 / 28, but 72x90x90 25.0 / 23.1, 40x130x130 27 / 26; nx odd 63x49x33 8.1 / 9.1, 73x90x90 level; FP32
// Smagorinsky 62x49x33 5.8 / 6.9, 120x90x90 0.92 of the time, 72x90x90 1.12.
template <class RS>
inline bool whole_rows(const StepArgs<RS>& a, int row, int idle, int nodes) {
    return (a.wall_mask & 60) && (long long)a.nx * a.ny * a.nzc <= nodes &&
           ((row + 31) / 32 * 32 - row) * (long long)a.ny * a.nzc <= idle;
}

// Step kernel selection: one node per thread (k_step), except 16-bit storage with nx even,
// which runs two x-adjacent nodes per thread in packed FP32-pair arithmetic
// (k_step_pair_seq, step_pair.cuh: the 16-bit step is issue-bound, and the shared pull and the
// pair instructions halve its arithmetic per node).  FP32 storage stays one node per thread: its
// step already runs at the HBM bound, and it keeps the delta form, whose FP32 rounding acts on
// the collision increment only; FP64 is bound by its arithmetic.
template <class L, class ST, int C, int F, bool FO>
cudaError_t launch_form(const StepArgs<typename Store<ST>::R>& a, cudaStream_t s) {
    dim3 g;
    if constexpr (sizeof(ST) == 2) {
        if (a.nx % 2 == 0) {
            dim3 b(128);
            NodeMap m = node_grid<2>(a, 128, 16, &g);
            if (whole_rows(a, a.nx / 2, 7 << 14, 1 << 21)) {
                m.nx.m = 0;
                lattice_grid(a.nx / 2, a.ny, a.nzc, &g, &b);
            }
            return launch_pdl(k_step_pair_seq<L, ST, C, F, FO>, g, b, s, a, m);
        }
    }
    // FP64 (bound by a pipe that each SM has its own share of): blocks of 64 spread a small lattice more
    // evenly over the SMs (32^3: 512 blocks over 152 SMs instead of 256)
    constexpr int T = sizeof(ST) == 8 ? 64 : 128;
    if constexpr (L::D == 2) {
        // FP64 rows that leave more than a 16th of their blocks idle go in node order, but for lattices of a few us: idle
        // threads are idle FP64 pipes, and of rows of 65 to 128 nodes every second block, and so every second SM, gets
        // little (us a step, Newtonian Yu, plain grid / node order: 66x1264 cavity 29 / 18, 96x400 12.0 / 9.0, 257x300 17.1 /
        // 14.9, but 67x67 6.0 / 6.7)
        if constexpr (sizeof(ST) == 8) {
            const NodeMap m = node_grid<1>(a, T, 16, &g);
            if (m.nx.m != 0 && (long long)a.nx * a.ny > (1 << 14))
                return launch_pdl(k_step<L, ST, C, F, FO, false>, g, dim3(T), s, a, m);
        }
        // FP32, the lightest step: the plain grid always (1000^2, 2% of the threads idle: 97.4 GLUPS against 92.1 in
        // node order)
        dim3 b;
        lattice_grid(a.nx, a.ny, a.nzc, &g, &b, T);
        return launch_pdl(k_step<L, ST, C, F, FO, true>, g, b, s, a, NodeMap{});
    } else {
        // rows that nearly fill their blocks keep the plain grid only where both buffers take at most 64 MB, half of L2
        // (us a step, plain grid / node order: 62 MB, 121x89x38 channel, FP32 Newtonian Chai 11.0 / 11.7, FP16 Smagorinsky
        // Yu 15.0 / 16.4; D3Q19 FP32 Smagorinsky Yu channel nx = 125 20 MB 6.9 / 7.5, 45 MB 9.9 / 10.3, 62 MB 12.4 / 12.3, but
        // 75 MB 14.3 / 13.1, 130 MB 27.3 / 25.7, 400 MB 74 / 68): beyond, blocks that start off a 128-byte line cost
        // more than the two divisions
        const bool small = 2LL * L::Q * a.stride * (int)sizeof(ST) <= (64LL << 20);
        dim3 b(T);
        NodeMap m = node_grid<1>(a, T, small ? 16 : 0, &g);
        if (sizeof(ST) != 8 && whole_rows(a, a.nx, sizeof(ST) == 2 ? 7 << 14 : 1 << 16, 1 << 20)) {
            m.nx.m = 0;
            lattice_grid(a.nx, a.ny, a.nzc, &g, &b);
        }
        return m.nx.m == 0 ? launch_pdl(k_step<L, ST, C, F, FO, true>, g, b, s, a, m)
                           : launch_pdl(k_step<L, ST, C, F, FO, false>, g, b, s, a, m);
    }
}

template <class L, class ST, int C, int F>
cudaError_t launch_step_cf(const StepArgs<typename Store<ST>::R>& a, int force, cudaStream_t s) {
    return force ? launch_form<L, ST, C, F, true>(a, s) : launch_form<L, ST, C, F, false>(a, s);
}

// EXTRA_CLOSURES: the power law and the two Smagorinsky variants (lagged, deviatoric) are
// instantiated (FP32 and FP64 storage); 16-bit storage builds Newtonian and Smagorinsky only.
template <class L, class ST, bool EXTRA_CLOSURES>
cudaError_t launch_step(const StepArgs<typename Store<ST>::R>& a, int closure, int formula, int force,
                        cudaStream_t s) {
    const bool yu = formula == F_YU;
    switch (closure) {
        case CL_NEWTON:
            // with fixed rates a step needs no S: 16-bit storage steps either formula by the shorter (Yu) moments,
            // FP32 and FP64 by their own, whose rounding differs (D2Q9 FP32 after 20 steps: Chai's 7.7e-8 from 64
            // bits, Yu's 9.5e-8)
            return yu || sizeof(ST) == 2 ? launch_step_cf<L, ST, CL_NEWTON, F_YU>(a, force, s)
                                         : launch_step_cf<L, ST, CL_NEWTON, sizeof(ST) == 2 ? F_YU : F_CHAI>(a, force, s);
        case CL_SMAG:
            return yu ? launch_step_cf<L, ST, CL_SMAG, F_YU>(a, force, s)
                      : launch_step_cf<L, ST, CL_SMAG, F_CHAI>(a, force, s);
        case CL_POWERLAW:
            if constexpr (EXTRA_CLOSURES)
                return yu ? launch_step_cf<L, ST, CL_POWERLAW, F_YU>(a, force, s)
                          : launch_step_cf<L, ST, CL_POWERLAW, F_CHAI>(a, force, s);
            return cudaErrorNotSupported;
        case CL_SMAG_LAGGED:
            if constexpr (EXTRA_CLOSURES)
                return yu ? launch_step_cf<L, ST, CL_SMAG_LAGGED, F_YU>(a, force, s)
                          : launch_step_cf<L, ST, CL_SMAG_LAGGED, F_CHAI>(a, force, s);
            return cudaErrorNotSupported;
        case CL_SMAG_DEV:
            if constexpr (EXTRA_CLOSURES)
                return yu ? launch_step_cf<L, ST, CL_SMAG_DEV, F_YU>(a, force, s)
                          : launch_step_cf<L, ST, CL_SMAG_DEV, F_CHAI>(a, force, s);
            return cudaErrorNotSupported;
        default:
            return cudaErrorInvalidValue;
    }
}

template <class L, class ST>
cudaError_t launch_init(const StepArgs<double>& a, int closure, const double* drho, const double* u, const double* gu,
                        const typename Store<ST>::R* ffield, typename Store<ST>::R* tau_field, cudaStream_t s) {
    constexpr int b = sizeof(ST) == 8 ? 64 : 128;
    const NodeMap m = node_map<1>(a);
    const dim3 g((unsigned)((m.threads + (long long)b - 1) / b));
    const InitConst<InitX<ST>> k = init_const<L, InitX<ST>>(a, closure);
    const InitConst<double> kd = init_const<L, double>(a, closure);
    if (ffield || a.F[0] != 0.0 || a.F[1] != 0.0 || a.F[2] != 0.0)
        k_init<L, ST, true><<<g, b, 0, s>>>(a, k, kd, m, drho, u, gu, ffield, tau_field);
    else
        k_init<L, ST, false><<<g, b, 0, s>>>(a, k, kd, m, drho, u, gu, ffield, tau_field);
    return cudaGetLastError();
}

}  // namespace lbm

#define LBM_DEFINE_ENTRY(TAG, L, ST, EXTRA_CLOSURES)                                                         \
    namespace lbm {                                                                                          \
    cudaError_t step_##TAG(const StepArgs<Store<ST>::R>& a, int closure, int formula, int force,             \
                           cudaStream_t s) {                                                                 \
        return launch_step<L, ST, EXTRA_CLOSURES>(a, closure, formula, force, s);                            \
    }                                                                                                        \
    cudaError_t init_##TAG(const StepArgs<double>& a, int closure, const double* drho, const double* u,      \
                           const double* gu, const Store<ST>::R* ffield, Store<ST>::R* tau_field,            \
                           cudaStream_t s) {                                                                 \
        return launch_init<L, ST>(a, closure, drho, u, gu, ffield, tau_field, s);                            \
    }                                                                                                        \
    }
