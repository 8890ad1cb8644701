// Instantiations of the small-tile kernels for FP16 inputs on the NVIDIA models (T-FDPA).
#include "mmasim_direct.cuh"
namespace mmasim { namespace direct {
cudaError_t launch_f16(const DevModel& m, const GemmArgs& g, DirectSize size, cudaStream_t st) {
    const bool h = m.rho == RHO_RNE_FP16;
    switch (m.L) {
        case 4: return h ? launch<FAM_T, fast::EK_F16, 4, RHO_RNE_FP16>(m, g, size, st) : launch<FAM_T, fast::EK_F16, 4, RHO_RZ_FP32>(m, g, size, st);
        case 8: return h ? launch<FAM_T, fast::EK_F16, 8, RHO_RNE_FP16>(m, g, size, st) : launch<FAM_T, fast::EK_F16, 8, RHO_RZ_FP32>(m, g, size, st);
        case 16: return h ? launch<FAM_T, fast::EK_F16, 16, RHO_RNE_FP16>(m, g, size, st) : launch<FAM_T, fast::EK_F16, 16, RHO_RZ_FP32>(m, g, size, st);
        default: return cudaErrorInvalidValue;
    }
}
}}
