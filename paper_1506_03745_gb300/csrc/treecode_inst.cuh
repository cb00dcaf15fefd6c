// Explicit instantiation and dispatch of the treecode kernels for one
// arithmetic type (included by treecode_f32.cu / treecode_f64.cu).
#include <algorithm>

#include "treecode.cuh"

namespace pgb {

template <typename real, int P>
static void launch_p(int stage, const UpArgs& up, const EvalArgs& ev, const void* xrel, void* mom, const void* far,
                     cudaStream_t s) {
    if (stage == PGB_STAGE_UPWARD) launch_upward<real, P>(up, mom, s);
    if (stage == STAGE_PANEL_MOMENTS) launch_panel_moments<real, P>(up, ev.n_pan, mom, s);
    if (stage == PGB_STAGE_P2P) launch_p2p<real>(ev, ev.K, xrel, s);
    if (stage == PGB_STAGE_M2P) launch_m2p<real, P>(ev, xrel, far, s);
}

}  // namespace pgb
