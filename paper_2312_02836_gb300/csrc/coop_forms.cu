// coop_forms.cu -- team kernels of two and four warps' sums and of the lane
// order (a translation unit of their own: they compile beside coop.cu's).
#include <cuda_runtime.h>

#include "coop_kernel.cuh"

const nb::TeamKernel nb::kOtherTeamKernels[nb::kOtherTeams] = {
    NB_TEAM(64, 64, 0, 64, 1),     NB_TEAM(64, 64, 1, 64, 1),
    NB_TEAM(256, 64, 1, 256, 1),   NB_TEAM(128, 128, 0, 128, 1),
    NB_TEAM(128, 128, 1, 128, 1),  NB_TEAM(256, 128, 1, 256, 1),
    NB_TEAM(32, 0, 1, 128, 2),     NB_TEAM(128, 0, 1, 128, 2),
};
