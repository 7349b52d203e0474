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

// Whether an FP32 two-buffer flow step on D3Q7 sets takes the TMA-staged kernel (given a phi field
// as scratch): rows of whole 16-byte pieces (a tensor copy's rule), the undivided lattice, no
// walls in x, and 30 million nodes, so that the tiles at the lattice's ends are few enough for
// what they cost more (512^3: 7.39 against 8.19 ms a step, 384^3: 3.20 against 3.46 ms, 256^3:
// 1.05 against 1.04 ms, 192^3: 0.49 against 0.44 ms).
inline bool flow_tma_applies(const DevParams& P) {
    return P.nx % 4 == 0 && P.nx >= 64 && P.ny >= 32 && P.n >= 30000000 && !P.wall_x && P.z_lo == 0 && P.z_hi == P.nz &&
           P.wall_zlo == P.wall_z && P.wall_zhi == P.wall_z;
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
