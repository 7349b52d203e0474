// Host-side launch interface between the C-ABI (lbm_abi.cu) and the per-storage kernel
// translation units (lbm_step_<type>.cu).
#pragma once

#include <cuda_runtime.h>

#include "lbm_device.cuh"

#define LBM_NFIELDS_DEV 10
#define LBM_NRED_DEV 10

namespace lbm {

struct FieldPtrs { void* p[LBM_NFIELDS_DEV]; };

// streaming modes (see lbm_kernels.cuh)
constexpr int kModeAAEven = 0, kModeAAOdd = 1, kModePull = 2;

// What a kernel whose bounded wait ran out leaves in the context's fault word.
constexpr unsigned kWaitFault = 0x57414954u;

constexpr int kBlockX = 128;

// Threads of a block of the per-node step and phi kernels, all of one row: 128, 96 or 64, whichever
// leaves the fewest lanes past the row's end; single warps in lattices so small that each SM gets at
// most two (512 x 8 FP64 couple: 5.2 us a step against 8.2). One row per block: with y the same for
// a whole block the wrap tests of Nbr stay uniform (two-row blocks cost the in-place FP16 step 6 %).
inline int step_width(int nx, long long nodes) {
    if (nodes <= 32 * 152 * 2) return 32;
    int bx = nx >= kBlockX ? kBlockX : (nx + 31) / 32 * 32;
    for (int b : {96, 64})
        if ((nx + b - 1) / b * b < (nx + bx - 1) / bx * bx) bx = b;
    return bx;
}

// Planes (rows, in 2D) a marching block goes through: the count, up to ``most``, for which the
// waves of blocks over the chip's ``slots`` times the planes each block computes, ``extra`` for
// the planes around the chunk among them, are fewest.
inline int march_chunk(long long tiles, int n, long long slots, double extra, int most = 32) {
    int best = 1;
    double cost = 1e300;
    for (int c = 1; c <= n && c <= most; ++c) {
        const long long blocks = tiles * ((n + c - 1) / c);
        const double t = double((blocks + slots - 1) / slots) * (c + extra);
        if (t <= cost) { cost = t; best = c; }
    }
    return best;
}

// 3D two-step kernel: a block of 32 x 16 threads, of which the inner 28 x 14 own nodes.
constexpr int T2X = 32, T2Y = 16, T2IX = T2X - 4, T2IY = T2Y - 2;
constexpr int kTwoStepsBlocks = 2;                                     // resident on an SM

// Whether two steps a pass take less time than single steps on a D3Q7 lattice without flow. A pass
// takes the time of the blocks' turns, their threads times the planes they compute, those past the
// box and around a chunk among them. A single step takes the longest of its memory traffic (less
// where the L2 holds the state), of its blocks' launches and of its lanes, idle ones among them. Both
// in ps a node and step, fitted to 130 boxes of 1 to 17 million nodes (two of them come out on the
// wrong side, by 1.5 %). Single step over
// two steps a pass, measured: 256^3 1.43, 128^3 1.29, 28x14x4000 2.04, 16x512x128 2.36, 64x64x4096
// 1.24, 150x84x80 1.01; below one, refused: 57x29x1000 0.85, 64x64x256 0.88, 101^3 0.95, 29x15x2400
// 0.68, 512x16x128 0.76, 1024x1024x1 0.65, 1024x1x1024 0.15.
inline bool two_steps_pay_3d(int nx, int ny, int nz) {
    const double n = double(nx) * ny * nz;
    const long long tiles = (long long)((nx + T2IX - 1) / T2IX) * ((ny + T2IY - 1) / T2IY), slots = 152 * kTwoStepsBlocks;
    const int zc = march_chunk(tiles, nz, slots, 2.0);
    const long long rounds = (tiles * ((nz + zc - 1) / zc) + slots - 1) / slots;
    const double turns = double(rounds) * slots * T2X * T2Y * (zc + 1.2) / n;
    const double pass = (n < 1.6e6 ? 5.0 : 3.5) + 8.9 * turns;
    const int bx = step_width(nx, (long long)n);
    const double rows = double(ny) * nz * ((nx + bx - 1) / bx) / n;    // blocks a node
    const double lanes = bx * rows;
    const double memory = 20.5 + 5.0 * (n < 1.1e6 ? 0.0 : (n < 1.4e6 ? (n - 1.1e6) / 0.3e6 : 1.0));
    double single = memory * (0.8 + 0.2 * lanes);
    for (double t : {1015.0 * rows, 17.5 * lanes})
        if (t > single) single = t;
    return pass <= single;
}

// 2D two-step kernel: warps, four to a block, of which the inner 28 lanes own nodes of a row.
constexpr int T2Warps = 4, kTwoSteps2DBlocks = 4;                      // resident on an SM

// Its grid: four windows of a row to a block and ``rows`` rows a chunk; folded, warps go on with the
// next chunk, where a quarter of them or more would have no window and there are rows enough to
// fill the chip (29x20000 D2Q9 30.1 -> 19.9 us a step, 120x2563 10.6 -> 8.2, 28x20000 22.8 -> 13.2).
// Elsewhere that is slower (384^2 4.8 -> 5.4, 29x200 1.9 -> 2.6): a row's addresses are then no longer
// the same for a whole block.
struct TwoSteps2D {
    int rows, bx, by, rounds;
    bool fold;
    TwoSteps2D(int nx, int ny) {
        const int wins = (nx + T2IX - 1) / T2IX, slots = 152 * kTwoSteps2DBlocks;
        bx = (wins + T2Warps - 1) / T2Warps;
        fold = 3 * T2Warps * bx >= 4 * wins && (long long)bx * ny > slots;
        rows = fold ? march_chunk(wins, ny, slots * T2Warps, 2.0) : march_chunk(bx, ny, slots, 2.0);
        by = (ny + rows - 1) / rows;
        if (fold) {
            bx = (wins * by + T2Warps - 1) / T2Warps;
            by = 1;
        }
        rounds = int(((long long)bx * by + slots - 1) / slots);
    }
};

// Whether two steps a pass take less time than single steps on an FP32 2D lattice without flow: yes,
// but for some lattices that the L2 holds, of rows of whole 128-byte lines, which a single step
// reads without a wasted byte. There by the rows a pass goes through, in us a step: single step over
// two steps a pass, D2Q9 64x4096 0.87, 256x2343 0.91, 384x1562 0.96 (refused), 512x781 1.09, 128x3125
// 1.05, 768^2 1.09; D2Q5 256x4687 0.88, 1024^2 0.96 (refused), 2048x512 1.03, 224x4464 1.06. All others of 220
// lattices, 16^2 to 4096^2 and from one column to one row, came out at 0.95 to 3.8.
inline bool two_steps_pay_2d(int nx, int ny, bool d2q9) {
    const double n = 1e-6 * nx * ny;
    if (nx % 32 || n < (d2q9 ? 0.2 : 0.95) || n > (d2q9 ? 0.7 : 1.4)) return true;
    const TwoSteps2D p(nx, ny);
    const double pass = p.rounds * (p.rows + 1.5) * (d2q9 ? 1.1 : 0.72);
    const int bx = step_width(nx, (long long)nx * ny);
    const double rows = 1.02e-3 * ny * ((nx + bx - 1) / bx);           // the launches of a single step's blocks
    return pass <= (d2q9 ? 2.0 + 19.4 * n : 1.9 + 10.8 * n) || pass <= rows;
}

// Whether an FP32 two-buffer flow step on D3Q7 sets takes the TMA-staged kernel (given a phi field
// as scratch): rows of whole 16-byte pieces (a tensor copy's rule), the undivided lattice, no
// walls in x, 30 million nodes (measured from there on), and tiles that are
// worth it: a column of 32 x 15 threads at an end in x takes 1.4 times as long as another. Threads
// a node weighted so, and the fused kernel's time over this one's: 512^3 1.08, 1.107 (MRT 1.046);
// 384^3 1.08, 1.060; 2048x128x128 1.07, 1.137 (MRT 1.078); 512x243x242 1.10, 1.082; 552x700x118 MRT
// 1.10, 1.047; 800x96x400 1.13, 1.070; 224x224x640 1.12, 0.990; 256x256x458 1.16, 0.991 (MRT 0.955);
// 216x284x741 MRT 1.16, 0.974; 128x2048x128 1.20, 0.907; 128x128x2048 1.27, 0.888; 64x700x671 1.41,
// 0.789; 1024x32x917 1.44, 0.884. In flat lattices the planes around a chunk weigh more: 2048x2048x8
// 1.045, 4096x2048x4 1.006 (MRT 0.970), 4096x4096x2 0.985.
inline bool flow_tma_applies(const DevParams& P) {
    if (!(P.nx % 4 == 0 && P.nx >= 64 && P.ny >= 32 && P.nz >= 8 && P.n >= 30000000 && !P.wall_x && P.z_lo == 0 &&
          P.z_hi == P.nz && P.wall_zlo == P.wall_z && P.wall_zhi == P.wall_z))
        return false;
    const int tx = (P.nx + 31) / 32, ty = (P.ny + 14) / 15;            // two of the tx columns stand at an end
    return 32.0 * 15.0 * (tx + 0.4 * 2) * ty <= (P.coll == 2 ? 1.09 : 1.13) * P.nx * P.ny;
}

#define LBM_DECLARE_LAUNCHERS(SUFFIX)                                                                   \
    void launch_init_##SUFFIX(const DevParams&, const StateView&, int lat, bool flow, bool pull,         \
                              const double*, const double*, const double*, cudaStream_t);                \
    void launch_phi_##SUFFIX(const DevParams&, const StateView&, int lat, int mode, void* phi,           \
                             cudaStream_t);                                                              \
    void launch_plane_phi_##SUFFIX(const DevParams&, const StateView&, int lat, int mode, int z, void* out, \
                                   cudaStream_t);                                                        \
    void launch_step_##SUFFIX(const DevParams&, const StateView&, const StateView&, int lat, bool flow, \
                              int mode, void* phi, cudaStream_t);                                        \
    void launch_two_steps_##SUFFIX(const DevParams&, const StateView&, const StateView&, int lat,        \
                                   unsigned* fault, cudaStream_t);                                        \
    void launch_fused_##SUFFIX(const DevParams&, const StateView&, const StateView&, void* phi_work,      \
                               unsigned* fault, cudaStream_t);                                           \
    void launch_fields_##SUFFIX(const DevParams&, const StateView&, int lat, bool flow, int mode,        \
                                void* phi, FieldPtrs, cudaStream_t);                                     \
    void launch_reduce_##SUFFIX(const DevParams&, const StateView&, int lat, bool flow, int mode,        \
                                void* phi, void* bits, double* partials, int nblocks, cudaStream_t);

void launch_adjoint_step(const DevParams&, const StateView&, int storage, int lat, bool odd, const void* lam_next,
                         void* lam, double* partials, cudaStream_t);
void launch_adjoint_seed(const DevParams&, const StateView&, int storage, int lat, bool odd, const void* phib,
                         const void* muAb, const void* muBb, void* lam, double* partials, cudaStream_t);
void launch_adjoint_init(const DevParams&, int storage, int lat, const double* phi0, const double* cA0,
                         const double* cB0, const void* lam, double* phi0b, double* partials, cudaStream_t);
void launch_theta_final(const double* partials, int rows, double* out, cudaStream_t);
long long adjoint_rows(const DevParams& P);
int adjoint_ntheta();

LBM_DECLARE_LAUNCHERS(f64)
LBM_DECLARE_LAUNCHERS(f32)
LBM_DECLARE_LAUNCHERS(f16)
LBM_DECLARE_LAUNCHERS(bf16)

}  // namespace lbm
