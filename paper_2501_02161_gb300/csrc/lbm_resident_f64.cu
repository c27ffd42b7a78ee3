// lbm_resident_f64.cu -- resident kernels of the 64-bit storage, in a
// translation unit of their own.
#include "lbm_dispatch.cuh"
#include "lbm_resident.cuh"

namespace lbm {

cudaError_t resident_flow_f64(int stencil, ResPhase ph, const FlowLaunch& a, const ResPlan& p, const ResWords& w,
                              int steps, cudaStream_t s) {
    const auto x = dispatch::flow_args<0>(a);
    if (stencil == 0) {
        if (ph == RP_FLOW) return launch_resident<ResFlow<D2Q9, double, double, double>>(x, p, w, steps, s);
        return launch_resident<ResAdjoint<D2Q9, double, double, false>>(x, p, w, steps, s);
    }
    if (ph == RP_FLOW) return launch_resident<ResFlow<D3Q19, double, double, double>>(x, p, w, steps, s);
    if (ph == RP_ADJ) return launch_resident<ResAdjoint<D3Q19, double, double, false>>(x, p, w, steps, s);
    return launch_resident<ResAdjoint<D3Q19, double, double, true>>(x, p, w, steps, s);
}

cudaError_t resident_thermal_f64(ResPhase ph, const ThermLaunch& a, const ResPlan& p, const ResWords& w,
                                 int steps, cudaStream_t s) {
    const auto x = dispatch::therm_args<0>(a);
    if (ph == RP_THERM) return launch_resident<ResHeat<double, double, double>>(x, p, w, steps, s);
    return launch_resident<ResHeatAdjoint<double, double>>(x, p, w, steps, s);
}

}  // namespace lbm
