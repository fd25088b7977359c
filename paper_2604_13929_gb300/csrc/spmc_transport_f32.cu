// spmc_transport_f32.cu -- FP32 transport kernels: the streamlined
// production kernel (spmc_transport_f32.cuh) and the float instantiations of
// the generic template (kept as variant 0 and for batched launches).
#include "spmc_transport_f32.cuh"

namespace spmc {

namespace {

using FastKernel = void (*)(TransportParams, BatchParams);

// The streamlined kernel of a launch.  Runs that record photons and volumes
// of 2^26 bricks and more take the builds with 64-bit voxel addresses,
// unwrapped positions and per-photon counts (mirror faces decided at run time
// there).
FastKernel fast_kernel(bool field, bool mirror, bool wide) {
    if (wide) return field ? &transport_f32_kernel<true, true, false, true> : &transport_f32_kernel<false, true, false, true>;
    if (mirror)
        return field ? &transport_f32_kernel<true, true, false, false> : &transport_f32_kernel<false, true, false, false>;
    return field ? &transport_f32_kernel<true, false, false, false> : &transport_f32_kernel<false, false, false, false>;
}

FastKernel fast_batch_kernel(bool mirror) {
    return mirror ? &transport_f32_kernel<true, true, true, false> : &transport_f32_kernel<true, false, true, false>;
}

size_t batch_smem(int threads) { return f32_smem(true, true, threads); }

const void *batch_kernel(int variant, bool mirror) {
    if (variant == 0) return reinterpret_cast<const void *>(&transport_kernel<float, true, true, true>);
    return reinterpret_cast<const void *>(fast_batch_kernel(mirror));
}

}  // namespace

const void *kernel_f32(bool field, bool mirror, int variant, bool wide) {
    return variant == 0 ? kernel_ptr<float>(field, mirror)
                        : reinterpret_cast<const void *>(fast_kernel(field, mirror, wide));
}

size_t smem_f32(bool field, int variant, int threads) {
    return variant == 0 ? 0 : f32_smem(field, false, threads);
}

cudaError_t launch_transport_f32(TransportParams p, bool field, int blocks, int threads,
                                 size_t smem, cudaStream_t s, const LaunchExtras &e) {
    if (e.variant == 0) return launch_transport<float>(p, field, blocks, threads, smem, s);
    // Photons by warp: 32 at the start (fewer, down to 8, when there are not
    // enough for every warp), then claims of 32 that shrink with the photons
    // per warp so that the last claims stay balanced.
    const u64 warps = (u64)blocks * (u64)(threads / 32), per_warp = p.n_photons / warps;
    p.first = per_warp >= 32 ? 32u : (per_warp < 8 ? 8u : (u32)per_warp);
    p.claim_base = warps * p.first;
    p.claim = per_warp >= 256 ? 32u : (per_warp < 64 ? 8u : (u32)(per_warp / 8));
    const BatchParams none{};
    fast_kernel(field, p.mirror != 0, e.wide)<<<blocks, threads, smem, s>>>(p, none);
    return cudaGetLastError();
}

cudaError_t occupancy_f32(bool field, bool mirror, int variant, bool wide, int threads, size_t smem,
                          int *blocks_per_sm) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, kernel_f32(field, mirror, variant, wide),
                                                         threads, smem);
}

// Batched launches: variant 0 the generic kernel (lanes of a warp carry
// photons of different problems), 1 the streamlined kernel (chunks of one
// problem per warp).  mirror: some problem has mirror lateral faces.
cudaError_t launch_transport_batch(BatchParams b, int variant, bool mirror, int blocks,
                                   int threads, cudaStream_t s) {
    TransportParams p{};
    p.compact_k = b.compact_k;
    const size_t smem = variant == 0 ? 0 : batch_smem(threads);
    if (variant == 0) transport_kernel<float, true, true, true><<<blocks, threads, 0, s>>>(p, b);
    else fast_batch_kernel(mirror)<<<blocks, threads, smem, s>>>(p, b);
    return cudaGetLastError();
}

cudaError_t occupancy_batch(int variant, bool mirror, int threads, int *blocks_per_sm) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, batch_kernel(variant, mirror),
                                                         threads, variant == 0 ? 0 : batch_smem(threads));
}

}  // namespace spmc
