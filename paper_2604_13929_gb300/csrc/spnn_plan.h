// spnn_plan.h -- launch rules of the surrogate's GEMM kernels as plain host
// functions (no CUDA), so that they can be checked without a device.
#pragma once

#include <cstdint>

namespace spnn {

// Shared-memory budget in bytes of a rows GEMM's stage ring.  Half an SM's (two
// CTAs, eight epilogue warps) by default; twice that for a CTA whose accumulators
// take all of TMEM and which therefore runs alone on its SM.  A launch of at most
// two output tiles (box x N tile) per SM may have most of an SM too: its CTAs run a
// tile or two, so the latency of their loads shows (U-Net of batch 1: 16^3 128 -> 128
// 30 -> 26 us, 256 -> 128 46 -> 38 us).  Not so with a scatter epilogue (up forward,
// down input gradient), which bounds those layers: up 8^3 256 -> 128 took 83 us at
// batch 64 with half an SM and 114 us with a whole one, down 16^3 128 -> 256 input
// gradients 110 and 144 us.
inline uint32_t ring_budget(long long tiles, int grid_n, int sms, bool scatter, bool alone, int option_kb) {
    if (option_kb > 0) return (uint32_t)option_kb * 1024u;
    if (alone) return 220u * 1024u;
    return !scatter && tiles * grid_n <= 2ll * sms ? 200u * 1024u : 110u * 1024u;
}

}  // namespace spnn
