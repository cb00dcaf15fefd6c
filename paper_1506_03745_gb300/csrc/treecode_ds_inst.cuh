// Launches of the double-single kernels for one order P (included by
// treecode_ds.cu for P 0..8 and treecode_ds_hi.cu for P 10, 12, 15, so that
// the two halves compile in parallel).
#pragma once
#include <algorithm>

#include "p2p_ds.cuh"

namespace pgb {

template <int P>
inline void launch_ds(int stage, const UpArgs& up, const EvalArgs& ev, const void* xrel, void* mom,
                      const void* far, cudaStream_t s) {
    // P2M and the moment shifts, then the far-field coefficients, all in
    // double-single on the FP32 pipe
    if (stage == PGB_STAGE_UPWARD) launch_upward<ds, P>(up, mom, s);
    if (stage == STAGE_PANEL_MOMENTS) launch_panel_moments<ds, P>(up, ev.n_pan, mom, s);
    if (stage == PGB_STAGE_P2P) launch_p2p_ds(ev, ev.K, xrel, s);
    if (stage == PGB_STAGE_M2P) launch_m2p<ds, P>(ev, xrel, far, s);
}

}  // namespace pgb
