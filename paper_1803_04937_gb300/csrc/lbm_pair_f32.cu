// Two D3Q19 steps per pass, FP32 storage (see lbm_pair.cuh).
#include "lbm_pair.cuh"

namespace lbm {

bool pair_runs_f32(const Geo &g, bool always, bool mrt, bool rho0_is_rho)
{
    return pair_runs<Lat19>(g, always, {mrt ? 3.1 : 2.8, 2.65, mrt && rho0_is_rho ? 1.0 : 0.3, 45.5});
}

cudaError_t launch_pair_f32(const void *src, void *dst, const Geo &g, const CollBoth &c, cudaStream_t s)
{
    const RelaxPacked p = to_packed(to_relax<float>(c));
    const PairPlanes<Lat19> S = pair_planes<Lat19>(src, g.ncell), D = pair_planes<Lat19>(dst, g.ncell);
    const bool walls = g.wall_x || g.wall_y || g.wall_z;
#define LBM_PAIR(R, W, M) return launch_pair_k<Lat19, R, W, M>(S, D, g, p, s)
    if (c.mrt) {
        if (c.rho0_is_rho) { if (walls) LBM_PAIR(true, true, true); LBM_PAIR(true, false, true); }
        if (walls) LBM_PAIR(false, true, true);
        LBM_PAIR(false, false, true);
    }
    if (c.rho0_is_rho) { if (walls) LBM_PAIR(true, true, false); LBM_PAIR(true, false, false); }
    if (walls) LBM_PAIR(false, true, false);
    LBM_PAIR(false, false, false);
#undef LBM_PAIR
}

}  // namespace lbm
