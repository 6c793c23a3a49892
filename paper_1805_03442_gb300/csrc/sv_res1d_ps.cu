// sv_res1d_ps.cu -- the resident 1D step loop (sv_res1d.cuh): perturbation layout.
#include "sv_res1d.cuh"

namespace sv {

void* res1d_pick_ps(const KParams& kp) { return res_pick<float, 3>(kp); }

}  // namespace sv
