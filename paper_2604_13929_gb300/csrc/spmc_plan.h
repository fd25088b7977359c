// spmc_plan.h -- launch rules of the transport kernels as plain host functions
// (no CUDA), so that they can be checked without a device.
#pragma once

#include <algorithm>
#include <cstddef>

namespace spmc {

// Voxel steps per pass of the streamlined FP32 kernel: the caller's value, or with
// 0 (automatic) the length that suits the optics.  A lane whose photon interacts
// waits for the end of the pass; with an interaction every 1.5 / (mu_s (1 - phi))
// steps or so, a pass of 8 wastes more than a second event phase costs below
// about 16 (16 masks of 64^3 36.1 -> 34.1 ms and 256^3 phi 0.70 profiles 58.5 ->
// 57.0 ms with 4; 256^3 phi 0.90, 30 steps, 40.6 -> 40.8 ms and keeps 8).
constexpr int kPassSteps = 8, kPassStepsDense = 4, kPassStepsMax = 64;
inline int pass_steps(int option, double mus, double porosity) {
    if (option > 0) return option;
    return mus * (1.0 - porosity) * 16.0 > 1.5 ? kPassStepsDense : kPassSteps;
}

// Mask bricks that a CTA stages when `want` are asked for (staging more or fewer
// changes no result).  The streamlined FP32 kernel's own shared memory, `own` bytes
// of tallies and lane state, comes out of the slab where the whole slab beside it
// would cost a resident CTA that a kernel with little more than its tallies keeps;
// `resident` CTAs fit an SM without a slab.  12288 bricks (96 KB, the automatic
// slab) with 256 threads: two CTAs need 11886 or fewer.  1e6 photons, depth profiles,
// one CTA -> two: 256^3 phi 0.90 20.7 -> 14.0 ms, phi 0.70 29.9 -> 21.1 ms.
constexpr size_t kSmemPerSm = 228 * 1024, kSmemPerCta = 227 * 1024, kSmemReserved = 1024, kSmemBare = 4352;
inline int staged_bricks(int want, size_t own, int resident) {
    const size_t slab = (size_t)want * 8;
    // too large for any kernel: left to the launch to refuse
    if (want <= 0 || !own || slab + kSmemBare > kSmemPerCta) return want;
    const int ctas = std::max(1, std::min(resident, (int)(kSmemPerSm / (slab + kSmemBare + kSmemReserved))));
    const size_t room = std::min(kSmemPerCta, kSmemPerSm / (size_t)ctas - kSmemReserved);
    return (int)(std::min(slab, room > own ? room - own : 0) / 8);
}

}  // namespace spmc
