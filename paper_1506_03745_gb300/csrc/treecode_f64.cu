// FP64 treecode kernels (P2M/M2M upward pass, fused P2P + M2P evaluation).
#include "treecode_inst.cuh"

namespace pgb {
void treecode_launch_f64(int stage, int P, const UpArgs& up, const EvalArgs& ev, const void* xrel, void* mom,
                         const void* far, cudaStream_t s) {
    switch (P) {
        case 0: launch_p<double, 0>(stage, up, ev, xrel, mom, far, s); break;
        case 1: launch_p<double, 1>(stage, up, ev, xrel, mom, far, s); break;
        case 2: launch_p<double, 2>(stage, up, ev, xrel, mom, far, s); break;
        case 3: launch_p<double, 3>(stage, up, ev, xrel, mom, far, s); break;
        case 4: launch_p<double, 4>(stage, up, ev, xrel, mom, far, s); break;
        case 5: launch_p<double, 5>(stage, up, ev, xrel, mom, far, s); break;
        case 6: launch_p<double, 6>(stage, up, ev, xrel, mom, far, s); break;
        case 7: launch_p<double, 7>(stage, up, ev, xrel, mom, far, s); break;
        case 8: launch_p<double, 8>(stage, up, ev, xrel, mom, far, s); break;
        case 10: launch_p<double, 10>(stage, up, ev, xrel, mom, far, s); break;
        case 12: launch_p<double, 12>(stage, up, ev, xrel, mom, far, s); break;
        case 15: launch_p<double, 15>(stage, up, ev, xrel, mom, far, s); break;
        default: fail(PGB_EINVAL, "P out of range");
    }
}

void near_build_f64(const EvalArgs& ev, int K, const void* ng, const void* xrel, void* mat, cudaStream_t s) {
    launch_near_build<double>(ev, K, ng, xrel, mat, s);
}
}  // namespace pgb
