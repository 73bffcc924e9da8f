// k_generic_d3.cu -- instantiations of the generic step kernel for D = 3.
#include "k_generic_step.cuh"

namespace lbmh {
cudaError_t step_generic_d3(const StepArgs &a, int blocks, int threads, cudaStream_t s) {
    switch (a.lat.P) {
    case lbmd::P_F64: return lbmd::launch_generic_dp<3, lbmd::P_F64>(a, blocks, threads, s);
    case lbmd::P_F32: return lbmd::launch_generic_dp<3, lbmd::P_F32>(a, blocks, threads, s);
    case lbmd::P_F16S: return lbmd::launch_generic_dp<3, lbmd::P_F16S>(a, blocks, threads, s);
    default: return cudaErrorInvalidValue;
    }
}

const void *small_kernel_d3(int P, int eq, int bulk, bool lanes, bool many) {
    if (lanes) return lbmd::lanes_kernel_d<3>(eq, bulk);
    switch (P) {
    case lbmd::P_F64: return lbmd::small_kernel_dp<3, lbmd::P_F64>(eq, bulk, many);
    case lbmd::P_F32: return lbmd::small_kernel_dp<3, lbmd::P_F32>(eq, bulk, many);
    case lbmd::P_F16S: return lbmd::small_kernel_dp<3, lbmd::P_F16S>(eq, bulk, many);
    default: return nullptr;
    }
}
}  // namespace lbmh
