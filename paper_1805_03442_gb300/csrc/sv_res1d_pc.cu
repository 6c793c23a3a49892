// sv_res1d_pc.cu -- the resident 1D step loop (sv_res1d.cuh): compensated pressure.
#include "sv_res1d.cuh"

namespace sv {

void* res1d_pick_pc(const KParams& kp) { return res_pick<float, 2>(kp); }

}  // namespace sv
