// spmc_plan.h -- launch rules of the transport kernels as plain host functions
// (no CUDA), so that they can be checked without a device.
#pragma once

namespace spmc {

// Voxel steps per pass of the streamlined FP32 kernel: the caller's value, or with
// 0 (automatic) the length that suits the optics.  A lane whose photon interacts
// waits for the end of the pass; with an interaction every 1.5 / (mu_s (1 - phi))
// steps or so, a pass of 8 wastes more than a second event phase costs below
// about 16 (16 masks of 64^3 36.1 -> 34.1 ms and 256^3 phi 0.70 profiles 58.5 ->
// 57.0 ms with 4; 256^3 phi 0.90, 30 steps, 40.6 -> 40.8 ms and keeps 8).
constexpr int kPassSteps = 8, kPassStepsDense = 4;
inline int pass_steps(int option, double mus, double porosity) {
    if (option > 0) return option;
    return mus * (1.0 - porosity) * 16.0 > 1.5 ? kPassStepsDense : kPassSteps;
}

}  // namespace spmc
