// k_chain_f64.cu -- coupled van der Pol chain kernels, one warp per system where the batch is small (oscillator g = q * 32 + lane);
// plain FP64 form; compiled without multiply-add contraction.
#include "run_model.cuh"

namespace bode {

cudaError_t launch_chain_team_f64(int method, int team, const RhsEntry& r, const BatchArgs& a, const LaunchCfg& c);

cudaError_t launch_chain_f64(int method, const RhsEntry& r, const BatchArgs& a, const LaunchCfg& c, bool* ok) {
    *ok = true;
    if (c.team == 0 && r.neq <= 128) {
        const int team = grid_team_f64(r.neq / 2, a.nsys, c.sm_count, true, method, a.index != nullptr);
        if (team < 32) return launch_chain_team_f64(method, team, r, a, c);
    }
    if (r.neq <= 64) return run_model_prec<ChainModel<32, 1>, ODE_PREC_FP64>(method, a, grid_ctx(r), c);
    if (r.neq <= 128) return run_model_prec<ChainModel<32, 2>, ODE_PREC_FP64>(method, a, grid_ctx(r), c);
    *ok = false;
    return cudaSuccess;
}

}  // namespace bode
