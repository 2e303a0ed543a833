// step_block.cuh -- BLOCK_STEPS steps of a D2Q9 lattice per launch, tile by tile in shared memory.
//
// One step per launch reads and writes every population once (72 B a node in FP32): from HBM that bounds large
// lattices (4096^2 at 95 GLUPS, the copy bandwidth), and a small lattice's step takes 3 us however little it
// computes (256^2 at 21.5 GLUPS).  Here a block owns BW x BH nodes and advances them 4 steps in one launch: the
// first step pulls from global memory and computes the tile with a margin of 3 nodes, each following step
// pulls from shared memory and computes a margin one node narrower, and the last one writes the tile's
// nodes to the destination buffer.  Margins are computed by every tile that needs them, so no block waits for
// another; a margin ends at a wall, where the pull reflects the node's own populations.  Every node update is
// the one-step kernel's, so the state equals one launch per step bit for bit.
//
// Tile: 32 x 20, so that the first step's 38 x 26 nodes take one pass of 1024 threads (1.27 node
// updates computed per one kept); 32 x 16 (1.31) where 32 x 20 leaves SMs without a tile.  Measured (Newtonian
// Yu, GLUPS per step launch / 32x16 / 32x20): 256^2 21.5 / 38.6 / 36.5, 512^2 56.9 / 72.7 / 75.8, 1000^2 98.9 /
// 104 / 110, 4096^2 95.3 / 122 / 131; 256 threads (several passes a step, few warps) 22 at 256^2, 110 at 4096^2;
// 64x32 120 at 4096^2, 6 steps 112, 2 steps 103 (32x16).  Where tiles are taken: block_pays.
//
// The bound keeps two blocks on an SM (32 registers).  Every form but the forced power law and the forced deviatoric
// closure takes 32 anyway; those took 42 to 47, one block a SM, and were slower than one launch per step (forced
// cavity 4096^2, us a step, one block / two / per step: deviatoric Yu 207 / 165 / 180, Chai 217 / 179 / 185; power
// law n = 0.5, 700^2 Yu 10.9 / 9.7 / 9.5, with 52 bytes spilled).
#pragma once

#include "launch.h"
#include "step.cuh"

namespace lbm {

constexpr int BW = 32, BLOCK_THREADS = 1024;
constexpr int BM = BLOCK_STEPS - 1;   // margin of the first step
constexpr int SW = BW + 2 * BM;       // width of the shared tile
// its height and its size, for tiles of BH rows
constexpr int tile_rows(int BH) { return BH + 2 * BM; }
constexpr int block_smem(int BH) { return 2 * 9 * SW * tile_rows(BH) * (int)sizeof(float); }

// Pull of the node (x, y) at tile position t of the shared populations s (population i at i * PITCH): periodic
// neighbours lie beside it in the tile, populations from behind a wall come from the node itself as in
// pull_general.
template <class L, int PITCH>
__device__ __forceinline__ void pull_tile(const StepArgs<float>& a, const float* s, int t, int x, int y,
                                          float (&f)[L::Q]) {
    const int w = a.wall_mask;
    const bool xl = (w & 1) && x == 0, xh = (w & 2) && x == a.nx - 1, yl = (w & 4) && y == 0,
               yh = (w & 8) && y == a.ny - 1;
    if (!(xl || xh || yl || yh)) {
        sfor<L::Q>([&](auto i) {
            f[i] = s[CV(i) * PITCH + t - L::c(CV(i), 0) - L::c(CV(i), 1) * SW];
        });
        return;
    }
    sfor<L::Q>([&](auto i) {
        constexpr int cx = L::c(CV(i), 0), cy = L::c(CV(i), 1);
        const bool ox = (cx > 0 && xl) || (cx < 0 && xh), oy = (cy > 0 && yl) || (cy < 0 && yh);
        if (!ox && !oy) {
            f[i] = s[CV(i) * PITCH + t - cx - cy * SW];
        } else {
            float v = s[opp<L>(CV(i)) * PITCH + t];
            const int face = ox ? (cx > 0 ? 0 : 1) : (cy > 0 ? 2 : 3);
            if (ox != oy && ((a.lid_mask >> face) & 1)) {
                const float cu = float(cx) * a.lid[face][0] + float(cy) * a.lid[face][1] + 0.0f * a.lid[face][2];
                v += float(double(6 * L::wnum(CV(i))) / L::WDEN) * a.rho0 * cu;
            }
            f[i] = v;
        }
    });
}

// Position p of a periodic axis of n nodes, wrapped.  A tile reaches less than its own extent beyond the lattice, so
// one step of n is enough unless the axis is shorter than that; a loop for every node instead cost more
// than the tiles gained on periodic lattices (4096^2 Newtonian Yu, 172 us a step with it, 139 without, 175 one by one).
template <int EXTENT>
__device__ __forceinline__ int wrap_pos(int p, int n) {
    if (n < EXTENT) return p < 0 ? n - 1 - (-1 - p) % n : p % n;
    return p < 0 ? p + n : (p >= n ? p - n : p);
}

template <class L, int CLOSURE, int FORMULA, bool FORCE, int BH>
__global__ void __launch_bounds__(BLOCK_THREADS, 2) k_step_block(const StepArgs<float> a) {
    constexpr int SH = tile_rows(BH), PITCH = SW * SH;
    extern __shared__ float sm[];
    pdl_wait();
    pdl_release();
    const int ox = blockIdx.x * BW - BM, oy = blockIdx.y * BH - BM;
    const bool wx = (a.wall_mask & 3) != 0, wy = (a.wall_mask & 12) != 0;
    sfor<BLOCK_STEPS>([&](auto k) {
        // step k computes the tile less k nodes on each side of the shared area
        constexpr int W = SW - 2 * CV(k), H = SH - 2 * CV(k);
        constexpr bool FIRST = CV(k) == 0, LAST = CV(k) == BLOCK_STEPS - 1;
        const float* from = sm + (CV(k) & 1 ? 0 : 1) * 9 * PITCH;
        float* to = sm + (CV(k) & 1) * 9 * PITCH;
        for (int t = threadIdx.x; t < W * H; t += BLOCK_THREADS) {
            const int ly = t / W + CV(k), lx = t - (t / W) * W + CV(k);
            const int x = wx ? ox + lx : wrap_pos<SW>(ox + lx, a.nx);
            const int y = wy ? oy + ly : wrap_pos<SH>(oy + ly, a.ny);
            bool mine = x >= 0 && x < a.nx && y >= 0 && y < a.ny;  // false only beyond a wall
            if (LAST) mine = mine && ox + lx < a.nx && oy + ly < a.ny;  // and past a ragged end
            if (!mine) continue;
            const int at = ly * SW + lx, node = y * a.nx + x;
            float f[L::Q];
            if constexpr (FIRST)
                pull<L, float>(a, x, y, 0, f);
            else
                pull_tile<L, PITCH>(a, from, at, x, y, f);
            if constexpr (LAST)
                step_body<L, float, CLOSURE, FORMULA, FORCE>(a, f, node);
            else
                collide<L, float, CLOSURE, FORMULA, FORCE>(
                    a, f, node, [&](auto i, float v) { to[CV(i) * PITCH + at] = v; });
        }
        if constexpr (!LAST) __syncthreads();
    });
}

// Whether tiles step the lattice faster than one launch per step does (sms: the device's SMs).  us a step, one by one /
// in tiles, Newtonian Yu and Smagorinsky Chai (N, S) unless named:
//  - Tiles that are all resident at once always do: a step launch takes 2.4 us or more (periodic 257x300 N 2.7 / 1.9, S
//    3.0 / 2.7; 3x6000 N 3.3 / 2.6; 6000x1 N 2.6 / 2.3 but S 2.5 / 2.9).
//  - Otherwise not where they compute a third more positions than the one-step grid: 20000x5 periodic S 3.1 / 6.3,
//    20000x41 cavity S 8.5 / 10.3, 20000x45 8.9 / 8.9, 65x20000 cavity N 21 / 20.
//  - Between walls they do at any size (700^2 N 6.7 / 5.5, S 7.9 / 7.4; 1000^2 10.3 / 9.3, 12.2 / 12.3; 4096^2 177 / 129,
//    182 / 164), except forced Smagorinsky flow above two waves of blocks (512^2 6.0 / 5.2, 1000^2 13.5 / 14.5,
//    4096^2 193 / 208).
//  - Periodic (or walled one way): the one-step grid has no branches at walls, and while both buffers stay in L2 it is the
//    faster above two waves: 600^2 N 4.5 / 3.9, S 5.3 / 5.0; 700^2 5.8 / 5.5, 6.5 / 7.1; 1000^2 9.3 / 9.5, 10.3 / 12.1.  From
//    HBM tiles pay again for the fixed rates and the deviatoric closure (2048^2 N 45.7 / 36.2, deviatoric Yu 45.9 /
//    39.9), not for the others (S 48.0 / 49.9).  L2 holds 129 MB; at 104 MB (1200^2) N 14.5 / 13.0.
//  - The power law is bound by its sweeps, which margins repeat: up to 2^19 nodes (cavity n = 0.5 Yu: 512^2 6.3 / 5.7,
//    1000^2 14.4 / 15.8, 4096^2 200 / 218), periodic up to one and a half waves (512^2 n = 0.6 5.7 / 5.4, 600^2 6.6 / 6.9).
//    With n = 1 it takes none (cavity Yu 1000^2 11.0 / 11.2, 4096^2 179 / 161, forced 190 / 180; periodic Chai 600^2
//    5.1 / 4.8, 1000^2 10.3 / 12.1, 4096^2 176 / 178).
inline bool block_pays(const StepArgs<float>& a, int closure, int force, int sms) {
    const long long N = (long long)a.nx * a.ny, tiles = (a.nx + BW - 1LL) / BW * ((a.ny + 19LL) / 20);
    const bool walls = (a.wall_mask & 3) && (a.wall_mask & 12);
    const bool from_hbm = 2LL * 9 * (int)sizeof(float) * a.stride > (96LL << 20);
    const bool sweeps = closure == CL_POWERLAW && a.pl_nm1 != 0.0f;
    if (sweeps && N > (1LL << 19)) return false;
    if (tiles <= 2LL * sms) return true;
    dim3 g, b;
    lattice_grid(a.nx, a.ny, 1, &g, &b);
    if (10 * tiles * BW * 20 > 13LL * g.x * b.x * g.y * b.y) return false;
    if (walls && !(closure == CL_SMAG && force)) return true;
    if (tiles <= (sweeps ? 3LL : 4LL) * sms) return true;
    return from_hbm && (closure == CL_NEWTON || closure == CL_SMAG_DEV);
}

// Either launches the tiles or (prepare) raises the kernel's shared-memory limit, which belongs to the current CUDA
// context and so is set by every lbm_step call that takes tiles
template <int C, int F, bool FO, int BH>
cudaError_t launch_block_tile(const StepArgs<float>& a, bool prepare, cudaStream_t s) {
    auto* k = k_step_block<D2Q9, C, F, FO, BH>;
    if (prepare) return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, block_smem(BH));
    const dim3 grid((a.nx + BW - 1) / BW, (a.ny + BH - 1) / BH);
    return launch_pdl_smem(k, grid, dim3(BLOCK_THREADS), block_smem(BH), s, a);
}
template <int C, int F, bool FO>
cudaError_t launch_block_form(const StepArgs<float>& a, int rows, bool prepare, cudaStream_t s) {
    return rows == 20 ? launch_block_tile<C, F, FO, 20>(a, prepare, s) : launch_block_tile<C, F, FO, 16>(a, prepare, s);
}

template <int C>
cudaError_t launch_block_c(const StepArgs<float>& a, int rows, int formula, int force, bool prepare, cudaStream_t s) {
    if (formula == F_YU)
        return force ? launch_block_form<C, F_YU, true>(a, rows, prepare, s)
                     : launch_block_form<C, F_YU, false>(a, rows, prepare, s);
    return force ? launch_block_form<C, F_CHAI, true>(a, rows, prepare, s)
                 : launch_block_form<C, F_CHAI, false>(a, rows, prepare, s);
}

}  // namespace lbm
