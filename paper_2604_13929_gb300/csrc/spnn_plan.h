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
// gradients 110 and 144 us.  But for one case: with two N tiles, the first one's CTAs
// (up to a box each) take the SMs' two slots before the second's, and with between
// 5/3 and 2 boxes per SM they leave it so few that those do nearly all its tiles.  If
// the tiles are short (one or two K-steps), one CTA per SM, so that the N tiles follow
// one another, is faster: up 32^3 64 -> 32 at batch 1 (256 boxes) 33 us against 29 us,
// 288 boxes 37 and 33 us; 248 boxes 30 and 32 us, 304 29 and 35 us.
inline uint32_t ring_budget(long long tiles, int grid_n, int ksteps, int sms, bool scatter, bool alone,
                            int option_kb) {
    if (option_kb > 0) return (uint32_t)option_kb * 1024u;
    if (alone) return 220u * 1024u;
    const bool whole = scatter ? grid_n == 2 && ksteps <= 2 && 3 * tiles >= 5ll * sms && tiles < 2ll * sms
                               : tiles * grid_n <= 2ll * sms;
    return (whole ? 200u : 110u) * 1024u;
}

// Input planes per stage of the z-walk: the most that divide zp + 2 into at
// least two stages of at most six.
constexpr int slab_zc(int zp) { return zp == 16 ? 6 : (zp == 8 ? 5 : (zp == 4 ? 3 : 2)); }

// Boxes and ring of the z-walk of a conv3 GEMM whose 128-voxel tiles (bx x by) lie
// in one z-plane, `columns` of them over D planes; zp = 0: the layer does not fit
// it.  It takes layers of n = 16, 32 or 64 output channels (3 n <= 256 columns in
// one MMA) whose weights stay resident in half of shared memory; above that the
// z-taps no longer share the A reads that bound them, or the ring gets too short.
// Of the depths that fit two buffers into TMEM it takes the cheapest: an MMA of
// N columns costs about max(N / 2, (128 + N) / 4) cycles (tensor rate, operand
// reads of 128 bytes a cycle), and the boxes go over the SMs in whole rounds.
struct SlabShape {
    int zp, stages;                 // output planes per box; stages of slab_zc(zp) input planes
    uint32_t w_bytes, stage_bytes;
};
inline SlabShape slab_shape(int bx, int by, long long columns, int D, int n, int kc_total, int sms) {
    const SlabShape none{0, 0, 0, 0};
    if ((n != 16 && n != 32 && n != 64) || 27 * kc_total * n * 16 > 112 * 1024) return none;
    auto mma = [&](int k) { const int N = k * n; return N / 2 > (128 + N) / 4 ? N / 2 : (128 + N) / 4; };
    SlabShape s = none;
    long long best_cost = 0;
    for (int zp = 2; zp <= 16 && zp <= D; zp *= 2) {
        if (2 * zp * n > 512) break;
        const long long rounds = (columns * (D / zp) + sms - 1) / sms;
        const long long cost = rounds * ((zp - 2) * mma(3) + 2 * mma(2) + 2 * mma(1));
        if (!s.zp || cost <= best_cost) s.zp = zp, best_cost = cost;
    }
    if (!s.zp) return none;
    // one CTA per SM (its accumulators take up to 512 TMEM columns)
    s.w_bytes = 27u * kc_total * n * 16u;
    s.stage_bytes = (uint32_t)(2 * slab_zc(s.zp) * (by + 2) * bx * 16);
    s.stages = (int)((220u * 1024u - s.w_bytes) / s.stage_bytes);
    if (s.stages > 8) s.stages = 8;
    return s.stages < 3 || s.stage_bytes % 128 ? none : s;
}

}  // namespace spnn
