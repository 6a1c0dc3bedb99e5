// rd_step19.h -- host-side declarations of the 19-point step kernels (the
// isotropic Laplacian of eqs. (3)-(4)), one step per launch, for the models
// without Cahn-Hilliard.
#pragma once

#include <stddef.h>

#include "rd_internal.h"

namespace rdk {

// Shared-memory ring of the 19-point kernel: planes q .. q+4 rotate through
// 5 slots; a slot holds (ty + 2) rows of kTileQ + 2 four-cell vectors of
// every field side by side (``mu_field``: one float field after the state's),
// and a guard vector at both ends.
constexpr int kRing19 = 5;
constexpr int kGuard19 = 16;
__host__ __device__ constexpr int row19_bytes(int nfields, int ebytes, bool mu_field) {
    return (kTileQ + 2) * 4 * (nfields * ebytes + (mu_field ? 4 : 0));
}
__host__ __device__ constexpr int plane19_bytes(int nfields, int ebytes, bool mu_field, int ty) {
    return (ty + 2) * row19_bytes(nfields, ebytes, mu_field) + 2 * kGuard19;
}
__host__ __device__ constexpr size_t smem19_pass_bytes(int nfields, int ebytes, bool mu_field,
                                                       int ty) {
    // the ring, then 96 halo fetch descriptors
    return (size_t)kRing19 * plane19_bytes(nfields, ebytes, mu_field, ty) + 96 * 16;
}
constexpr size_t smem19_bytes(int nspecies, int ebytes, int ty) {
    return smem19_pass_bytes(nspecies, ebytes, false, ty);
}
inline int threads19(int ty) { return kTileQ * ty + 32; }

// Single-instance launchers (one translation unit per model).  With
// occ != nullptr they only report the CTAs per SM.
cudaError_t launch19_diffusion(int storage, const LaunchArgs& a, int grid, size_t smem,
                               cudaStream_t st, int* occ);
cudaError_t launch19_brusselator(int storage, const LaunchArgs& a, int grid, size_t smem,
                                 cudaStream_t st, int* occ);
cudaError_t launch19_air(int storage, const LaunchArgs& a, int grid, size_t smem,
                         cudaStream_t st, int* occ);
// The two launches of a 19-point Cahn-Hilliard step (pass 1: mu, pass 2: the
// update); ``smem`` is the larger of the two passes' needs (smem19_ch_bytes).
cudaError_t launch19_ch_front(int storage, int pass, const LaunchArgs& a, int grid, size_t smem,
                              cudaStream_t st, int* occ);
cudaError_t launch19_ch_table1(int storage, int pass, const LaunchArgs& a, int grid, size_t smem,
                               cudaStream_t st, int* occ);
inline size_t smem19_ch_bytes(int ebytes, int ty) {
    return smem19_pass_bytes(3, ebytes, true, ty);
}

}  // namespace rdk
