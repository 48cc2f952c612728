// step_unit.cu -- the single-cavity kernels at the paper's unit higher-order rates
// (collide_unit.cuh), compiled apart from the general form (step.cu).
#include "step_kernels.cuh"

namespace lbm {

template <typename S>
cudaError_t launch_step_unit(const DevState& s, int cur, const ParamsOf<S>& p, cudaStream_t st) {
    return launch_step_as<S, true>(s, cur, p, st);
}

template cudaError_t launch_step_unit<double>(const DevState&, int, const ParamsOf<double>&, cudaStream_t);
template cudaError_t launch_step_unit<float>(const DevState&, int, const ParamsOf<float>&, cudaStream_t);
template cudaError_t launch_step_unit<__half>(const DevState&, int, const ParamsOf<__half>&, cudaStream_t);
template cudaError_t launch_step_unit<__nv_bfloat16>(const DevState&, int,
                                                     const ParamsOf<__nv_bfloat16>&, cudaStream_t);

template <typename S>
bool step_imposable(const DevState& s, const ParamsOf<S>& p) {
    return !Storage<S>::deviation && has_unit_rates(p, s.Q) && cavity_kernel_fits(p);
}

template <typename S>
cudaError_t launch_step_imposed(const DevState& s, int cur, const ParamsOf<S>& p, const ImposedFields& imposed,
                                cudaStream_t st) {
    if constexpr (Storage<S>::deviation) return cudaErrorNotSupported;
    else return launch_step_imposed_as<S>(s, cur, p, imposed, st);
}

#define LBM_INSTANTIATE_IMPOSED(S)                                                                  \
    template bool step_imposable<S>(const DevState&, const ParamsOf<S>&);                            \
    template cudaError_t launch_step_imposed<S>(const DevState&, int, const ParamsOf<S>&,            \
                                                const ImposedFields&, cudaStream_t);
LBM_INSTANTIATE_IMPOSED(double)
LBM_INSTANTIATE_IMPOSED(float)
LBM_INSTANTIATE_IMPOSED(__half)
LBM_INSTANTIATE_IMPOSED(__nv_bfloat16)

}  // namespace lbm
