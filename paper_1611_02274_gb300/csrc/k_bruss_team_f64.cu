// k_bruss_team_f64.cu -- Brusselator grids with several systems per warp (four points a
// lane); plain FP64 form;
// compiled without multiply-add contraction.  grid_team_f64 (launch.cuh)
// chooses between these and the warp-per-system kernels.
#include "run_model.cuh"

namespace bode {

cudaError_t launch_bruss_team_f64(int method, int team, const RhsEntry& r, const BatchArgs& a, const LaunchCfg& c) {
    const GridCtx g = grid_ctx(r);
    switch (team) {
    case 1: return run_model_prec<BrussModel<1, 4>, ODE_PREC_FP64>(method, a, g, c);
    case 2: return run_model_prec<BrussModel<2, 4>, ODE_PREC_FP64>(method, a, g, c);
    case 4: return run_model_prec<BrussModel<4, 4>, ODE_PREC_FP64>(method, a, g, c);
    case 8: return run_model_prec<BrussModel<8, 4>, ODE_PREC_FP64>(method, a, g, c);
    default: return run_model_prec<BrussModel<16, 4>, ODE_PREC_FP64>(method, a, g, c);
    }
}

}  // namespace bode
