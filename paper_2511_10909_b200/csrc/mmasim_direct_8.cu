// Instantiations of the small-tile kernels for 8-bit inputs: T-FDPA with F = 13 and F = 25, ST-FDPA.
#include "mmasim_direct.cuh"
namespace mmasim { namespace direct {
cudaError_t launch_lut8(const DevModel& m, const GemmArgs& g, DirectSize size, cudaStream_t st) {
    if (g.redo) return launch_rest<FAM_ST, fast::EK_LUT8, 32, RHO_RZ_FP32>(m, g, st);
    if (m.family == FAM_ST) return launch<FAM_ST, fast::EK_LUT8, 32, RHO_RZ_FP32>(m, g, size, st);
    if (m.L == 16) {
        if (m.rho == RHO_RZ_E8M13) return launch<FAM_T, fast::EK_LUT8, 16, RHO_RZ_E8M13>(m, g, size, st);
        if (m.rho == RHO_RNE_FP16) return launch<FAM_T, fast::EK_LUT8, 16, RHO_RNE_FP16>(m, g, size, st);
    } else if (m.L == 32) {
        if (m.rho == RHO_RZ_E8M13) return launch<FAM_T, fast::EK_LUT8, 32, RHO_RZ_E8M13>(m, g, size, st);
        if (m.rho == RHO_RZ_FP32) return launch<FAM_T, fast::EK_LUT8, 32, RHO_RZ_FP32>(m, g, size, st);
        if (m.rho == RHO_RNE_FP16) return launch<FAM_T, fast::EK_LUT8, 32, RHO_RNE_FP16>(m, g, size, st);
    }
    return cudaErrorInvalidValue;
}
}}
