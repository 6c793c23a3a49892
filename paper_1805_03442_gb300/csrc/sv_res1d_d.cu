// sv_res1d_d.cu -- the resident 1D step loop (sv_res1d.cuh): double.
#include "sv_res1d.cuh"

namespace sv {

void* res1d_pick_d(const KParams& kp) { return res_pick<double, 0>(kp); }

}  // namespace sv
