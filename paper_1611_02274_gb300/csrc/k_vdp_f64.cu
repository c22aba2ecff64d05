// k_vdp_f64.cu -- van der Pol kernels (one thread per system, two for
// batches that leave sub-partitions idle); plain FP64 form; compiled without multiply-add contraction.
#include "run_model.cuh"

namespace bode {

cudaError_t launch_vdp_f64(int method, const RhsEntry&, const BatchArgs& a, const LaunchCfg& c, bool* ok) {
    *ok = true;
    // Two lanes a system while the doubled warps still fit the sub-partitions
    // one each: a step is then 178 FP64 instructions' time instead of 241,
    // past that twice the warps cost more than the shorter step gives.
    // Measured, one lane / two (with
    // 128- and 32-thread blocks): 100 systems 3.67 / 3.05 ms, 4,096 systems
    // 3.82 / 3.12; 12,000 systems keep one lane, 3.53.
    if (2 * a.nsys <= 32 * 4 * (int64_t)c.sm_count)
        return run_model_prec<VdpPairModel, ODE_PREC_FP64>(method, a, NoCtx{}, c);
    return run_model_prec<VdpModel, ODE_PREC_FP64>(method, a, NoCtx{}, c);
}

}  // namespace bode
