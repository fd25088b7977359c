// spnn_gemm.cu -- the tensor-core GEMM kernels of the surrogate: rows_kernel
// and slab_kernel (forward and input-gradient layers), wgrad_kernel,
// wgrad_halo_kernel and wgrad_rows_kernel (weight gradients).
//
// All are warp-specialised, 192 threads (slab_kernel 320):
//   warp 0      TMA producer: fills a ring of shared-memory stages,
//   warp 1      allocates TMEM and issues tcgen05.mma,
//   warps 2..5  epilogue: tcgen05.ld of the FP32 accumulators, fused
//               bias / residual / ReLU / ReLU-derivative mask, BF16 stores
//               (FP32 atomics for weight gradients).
// The MMA warp (and the weight-gradient producers) walk their K loop with all
// 32 lanes so that descriptor and coordinate arithmetic stays warp-uniform; one
// elected lane issues.  K loops carry their stage index and tile origin as
// running values: integer division per step costs a lone thread hundreds of
// cycles.  Stages hand over with mbarriers: "full" completes when TMA bytes
// land, "empty" when the MMAs that read the stage retire (tcgen05.commit).
// Every wait is bounded by kWaitLimitNs; a timeout sets an error flag, and the
// CTA still releases its TMEM and exits.
#include "spnn_internal.cuh"
#include "spnn_umma.cuh"

namespace spnn {

__device__ __forceinline__ uint8_t* align1024(uint8_t* p) {
    return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~uintptr_t(1023));
}

// Stage index and wrap count of a ring of S stages, advanced once per K-step
// (the K loops avoid integer division, which costs a lone thread hundreds of
// cycles per step).
struct Ring {
    int s = 0;
    uint32_t r = 0;
    __device__ __forceinline__ void next(int S) {
        if (++s == S) {
            s = 0;
            ++r;
        }
    }
};

// Origin of the tile after (x0, y0, z0, b0): the increment of tile_origin.
__device__ __forceinline__ void tile_next(const TileGrid& g, int& x0, int& y0, int& z0, int& b0) {
    if ((x0 += g.bx) < g.nx * g.bx) return;
    x0 = 0;
    if ((y0 += g.by) < g.ny * g.by) return;
    y0 = 0;
    if ((z0 += g.bz) < g.nz * g.bz) return;
    z0 = 0;
    b0 += g.bb;
}

// 16 channels of one voxel: 8 at p[0..7] and 8 one chunk plane further.
__device__ __forceinline__ void load16_planes(const __nv_bfloat16* p, long long plane, float (&f)[16]) {
    uint4 u[2] = {*reinterpret_cast<const uint4*>(p), *reinterpret_cast<const uint4*>(p + plane)};
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(u);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        float2 t = __bfloat1622float2(h[i]);
        f[2 * i] = t.x;
        f[2 * i + 1] = t.y;
    }
}

// TMA box of chunk plane c8: chunk-plane map (8x, y, z, b, c8) or stride-2 view (0, x, y, z, c8 B + b).
__device__ __forceinline__ void load_box(uint32_t dst, const CUtensorMap* m, uint32_t bar, bool strided, int c8,
                                         int x, int y, int z, int b, int B) {
    if (strided)
        tma_load_5d(dst, m, bar, 0, x, y, z, c8 * B + b);
    else
        tma_load_5d(dst, m, bar, 8 * x, y, z, b, c8);
}

// The MMAs of one conv3 K-step: nine (dz, dy) taps x EH K-slices of 16
// channels x MT subtiles.  Descriptors are the step's base descriptors plus
// start-address offsets in 16-byte units (no carry: every address is inside
// shared memory): tap_off[t9] for the tap, a_koff per K-slice, 128 (2048
// bytes) per subtile; B holds [slice][tap] blocks of n_tile rows.  Unrolled so
// that one instruction stream issues every MMA back to back.
template <int MT, int EH>
__device__ __forceinline__ void issue_conv_step(uint32_t tmem, uint64_t adesc, uint64_t bdesc,
                                                const uint32_t (&tap_off)[9], uint32_t a_koff, uint32_t n_tile,
                                                uint32_t idesc, bool first) {
#pragma unroll
    for (int t9 = 0; t9 < 9; ++t9)
#pragma unroll
        for (int i = 0; i < EH; ++i) {
            const uint64_t bd = bdesc + (uint64_t)((uint32_t)(2 * i * 9 + t9) * n_tile);
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                const uint64_t ad = adesc + (uint64_t)(tap_off[t9] + (uint32_t)i * a_koff + 128u * m);
                umma_bf16(tmem + (uint32_t)m * n_tile, ad, bd, idesc, (first && t9 == 0 && i == 0) ? 0u : 1u);
            }
        }
}

__device__ __forceinline__ void issue_conv_step(int mt, int eh, uint32_t tmem, uint64_t adesc, uint64_t bdesc,
                                                const uint32_t (&tap_off)[9], uint32_t a_koff, uint32_t n_tile,
                                                uint32_t idesc, bool first) {
    if (mt == 4 && eh == 2)
        issue_conv_step<4, 2>(tmem, adesc, bdesc, tap_off, a_koff, n_tile, idesc, first);
    else if (mt == 4)
        issue_conv_step<4, 1>(tmem, adesc, bdesc, tap_off, a_koff, n_tile, idesc, first);
    else if (mt == 2 && eh == 2)
        issue_conv_step<2, 2>(tmem, adesc, bdesc, tap_off, a_koff, n_tile, idesc, first);
    else if (mt == 2)
        issue_conv_step<2, 1>(tmem, adesc, bdesc, tap_off, a_koff, n_tile, idesc, first);
    else if (eh == 2)
        issue_conv_step<1, 2>(tmem, adesc, bdesc, tap_off, a_koff, n_tile, idesc, first);
    else
        issue_conv_step<1, 1>(tmem, adesc, bdesc, tap_off, a_koff, n_tile, idesc, first);
}

// ------------------------------------------------------------------------
// Rows GEMM (forward, input-gradient and transposed-conv layers).
// A tile: kc_step chunk planes of 128 rows x 16 bytes (2 KB each), K-major;
// B tile: kc_step planes of n_tile rows x 16 bytes, K-major.
//
// Persistent, dynamically scheduled: the producer claims the next tile from a
// global counter (so any grid size is safe: a CTA that becomes resident only
// after the others have claimed every tile finds none and exits; tiles are
// claimed in grid order) and hands its index to the MMA and epilogue warps
// through a ring of four shared slots (tile_full / tile_empty; index -1 ends
// the CTA).  The stage ring runs on
// across tiles, so the next tile's operands load while the current one
// multiplies.  The accumulators of consecutive tiles alternate
// between two TMEM buffers (nbuf = 2 when they fit in 512 columns): the
// epilogue of tile i reads one buffer while the MMAs of tile i + 1 fill the
// other.  acc_full[b] completes when the MMAs of a tile retire
// (tcgen05.commit), acc_empty[b] when the four epilogue warps have read it.
// ------------------------------------------------------------------------

// Origin of tile t (32-bit: a lone thread divides once per tile).
__device__ __forceinline__ void tile_origin_u32(const TileGrid& g, uint32_t t, int& x0, int& y0, int& z0,
                                                int& b0) {
    uint32_t q = t / (uint32_t)g.nx;
    x0 = (int)(t - q * (uint32_t)g.nx) * g.bx;
    t = q;
    q = t / (uint32_t)g.ny;
    y0 = (int)(t - q * (uint32_t)g.ny) * g.by;
    t = q;
    q = t / (uint32_t)g.nz;
    z0 = (int)(t - q * (uint32_t)g.nz) * g.bz;
    b0 = (int)q * g.bb;
}

// Epilogue of 16 accumulator columns of one voxel: bias, residual, ReLU or
// ReLU-derivative mask, two 16-byte BF16 stores (channels ch0 .. ch0 + 15 at
// off); adds the rounded outputs' dot product with head_w (if given) to head.
// mk: the two mask words, where the caller has loaded them already.
__device__ __forceinline__ void emit16(const EpiDest& d, const uint32_t (&v)[16], int ch0, long long off,
                                       const float* head_w, float& head, const uint4* mk = nullptr) {
    float f[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) f[i] = __uint_as_float(v[i]);
    if (d.bias) {
#pragma unroll
        for (int i = 0; i < 16; ++i) f[i] += d.bias[ch0 + i];
    }
    if (d.addend) {
        float a[16];
        load16_planes(d.addend + off, d.plane, a);
#pragma unroll
        for (int i = 0; i < 16; ++i) f[i] += a[i];
    }
    if (d.relu) {
#pragma unroll
        for (int i = 0; i < 16; ++i) f[i] = fmaxf(f[i], 0.f);
    }
    if (d.mask) {
        uint4 u[2];
        u[0] = mk ? mk[0] : *reinterpret_cast<const uint4*>(d.mask + off);
        u[1] = mk ? mk[1] : *reinterpret_cast<const uint4*>(d.mask + off + d.plane);
        const __nv_bfloat162* m = reinterpret_cast<const __nv_bfloat162*>(u);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float2 t = __bfloat1622float2(m[i]);
            f[2 * i] = (t.x > 0.f) ? f[2 * i] : 0.f;
            f[2 * i + 1] = (t.y > 0.f) ? f[2 * i + 1] : 0.f;
        }
    }
    uint4 w[2];
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(w);
#pragma unroll
    for (int i = 0; i < 8; ++i) h[i] = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
    *reinterpret_cast<uint4*>(d.out + off) = w[0];
    *reinterpret_cast<uint4*>(d.out + off + d.plane) = w[1];
    if (head_w) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float2 rb = __bfloat1622float2(h[i]);
            head += rb.x * head_w[ch0 + 2 * i] + rb.y * head_w[ch0 + 2 * i + 1];
        }
    }
}

// The MMAs of one stage (ZC input planes) of the z-walk, as one straight run of
// 3 ZC instructions: an input plane is only three MMAs of 48 to 96 cycles, and a
// loop that works out its operands takes a lone warp about 300 cycles a plane.
// So everything but the stage's bases is a compile-time constant: N output
// channels, START / END (the stage holds the box's first / last input planes,
// which feed fewer output planes), FIRST (the first K-step: the newest output
// plane of an MMA, its last N columns, is overwritten, in an MMA of its own).
// a: descriptor low word of the stage's first plane, zrow / row: 16-byte units
// of a z-plane and a y-row; b: low word of the K-step's weights; col: columns
// of output plane z - 1 of the stage's first input plane z (0 with START).
template <int N, int ZC, bool START, bool END, bool FIRST>
__device__ __forceinline__ void slab_stage(uint32_t col, uint32_t a, uint32_t a_hi, uint32_t zrow, uint32_t row,
                                           uint32_t b, uint32_t b_hi) {
#pragma unroll
    for (int zi = 0; zi < ZC; ++zi) {
        // output planes j0 <= j < j1 of (z - 1, z, z + 1)
        const int j0 = START ? (zi == 0 ? 2 : (zi == 1 ? 1 : 0)) : 0;
        const int j1 = END ? (zi == ZC - 1 ? 1 : (zi == ZC - 2 ? 2 : 3)) : 3;
        const int cnt = j1 - j0;
        const uint32_t c = col + (uint32_t)((START ? (zi < 2 ? 0 : zi - 2) : zi) * N);
        const uint32_t az = a + (uint32_t)zi * zrow, bz = b + (uint32_t)(j0 * N);
        if (FIRST && j1 == 3) {
            if (cnt > 1) umma_bf16_lo<1>(c, az, a_hi, bz, b_hi, idesc_bf16(128, (cnt - 1) * N, 0, 0));
            umma_bf16_lo<0>(c + (uint32_t)((cnt - 1) * N), az, a_hi, bz + (uint32_t)((cnt - 1) * N), b_hi,
                            idesc_bf16(128, N, 0, 0));
        } else {
            umma_bf16_lo<1>(c, az, a_hi, bz, b_hi, idesc_bf16(128, cnt * N, 0, 0));
        }
        umma_bf16_lo<1>(c, az + row, a_hi, bz + 3u * N, b_hi, idesc_bf16(128, cnt * N, 0, 0));
        umma_bf16_lo<1>(c, az + 2u * row, a_hi, bz + 6u * N, b_hi, idesc_bf16(128, cnt * N, 0, 0));
    }
}

// MMA warp of slab_kernel: the whole warp walks the K-steps, one elected lane
// issues (see rows_kernel).  ZST stages of ZC input planes per K-step.
template <int N, int ZC, int ZST>
__device__ __forceinline__ void slab_issue(const SlabParams& p, uint32_t bar0, uint32_t acc_full, uint32_t acc_empty,
                                           uint32_t w_full, uint32_t wbase, uint32_t sbase, uint32_t tmem) {
    const bool leader = elect_one();
    const int S = p.stages, ksteps = 3 * (p.kc_total / 2);
    const uint32_t acc_cols = (uint32_t)p.zp * N;
    const uint32_t row = (uint32_t)p.g.bx, zrow = row * (uint32_t)(p.g.by + 2);
    const uint64_t ad = smem_desc(sbase, zrow * 16u * ZC, 128), bd = smem_desc(wbase, 9u * N * 16u, 128);
    const uint32_t a_hi = (uint32_t)(ad >> 32), b_hi = (uint32_t)(bd >> 32), stage_u = p.stage_bytes / 16u;
    auto wait = [&](uint32_t bar, uint32_t parity) -> bool {
        const bool ok = __all_sync(0xffffffffu, mbar_wait(bar, parity, kWaitLimitNs));
        if (!ok && leader) atomicOr(p.err, ERR_TIMEOUT);
        return ok;
    };
    if (!wait(w_full, 0)) return;
    Ring q;
    uint32_t it = 0;
    for (int t = blockIdx.x; t < p.tiles; t += gridDim.x, ++it) {
        const uint32_t buf = it & 1u, use = it >> 1;
        if (use > 0 && !wait(acc_empty + 8u * buf, (use - 1) & 1u)) return;
        tc_fence_after();
        const uint32_t acc = tmem + buf * acc_cols;
        uint32_t b = (uint32_t)bd;
        for (int k = 0; k < ksteps; ++k, b += 18u * N) {       // (x-shift, pair of chunk planes)
#pragma unroll
            for (int st = 0; st < ZST; ++st, q.next(S)) {
                if (!wait(bar0 + 8u * q.s, q.r & 1u)) return;
                tc_fence_after();
                const uint32_t a = (uint32_t)ad + (uint32_t)q.s * stage_u;
                // the stage's first input plane is st ZC - 1
                const uint32_t col = acc + (uint32_t)(st == 0 ? 0 : (st * ZC - 2) * N);
                if (leader) {
                    if (st == 0) {
                        if (k == 0) slab_stage<N, ZC, true, false, true>(col, a, a_hi, zrow, row, b, b_hi);
                        else slab_stage<N, ZC, true, false, false>(col, a, a_hi, zrow, row, b, b_hi);
                    } else if (st == ZST - 1) {
                        if (k == 0) slab_stage<N, ZC, false, true, true>(col, a, a_hi, zrow, row, b, b_hi);
                        else slab_stage<N, ZC, false, true, false>(col, a, a_hi, zrow, row, b, b_hi);
                    } else {
                        if (k == 0) slab_stage<N, ZC, false, false, true>(col, a, a_hi, zrow, row, b, b_hi);
                        else slab_stage<N, ZC, false, false, false>(col, a, a_hi, zrow, row, b, b_hi);
                    }
                    umma_commit(bar0 + 8u * (S + q.s));
                }
                __syncwarp();
            }
        }
        if (leader) umma_commit(acc_full + 8u * buf);
        __syncwarp();
    }
}

// ------------------------------------------------------------------------
// conv3 walked along z (see SlabParams): warp 0 loads, warp 1 issues, eight
// epilogue warps.  Tiles go round-robin over the CTAs (every tile is the same
// work, one CTA per SM), their accumulators alternate between two TMEM buffers.
// K order per output: x-shift, pair of chunk planes, z-tap, y-tap, 16 channels
// -- the order of rows_kernel, so both give the same bits.  The first product
// of an output plane (z-tap -1 of the first K-step) overwrites while the two
// older planes of the same MMA accumulate: there the MMA is split in two.
//
// The rows kernel's MMAs of N = 16 and 32 columns are bound by their shared-
// memory reads (128 A rows each); with N = 3 n they come near the tensor rate
// (N = 96: 56 cycles of reads for 48 of arithmetic, three taps).  Measured, rows
// kernel -> this, batch 16 at 64^3, forward: 16 -> 32 channels 183 -> 115 us,
// 32 -> 32 301 -> 178 us (1.30 PFLOP/s), 64 -> 32 561 -> 356 us; input gradient:
// 32 -> 32 with mask 318 -> 199 us, 32 -> 64 349 -> 270 us (1.72 PFLOP/s).
// ------------------------------------------------------------------------
template <int N, int ZC, int ZST>
__global__ void __launch_bounds__(kSlabThreads, 1) slab_kernel(const __grid_constant__ SlabParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    const int S = p.stages;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + p.w_bytes + (size_t)S * p.stage_bytes);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S + 5);
    const uint32_t wbase = smem_u32(smem), sbase = wbase + p.w_bytes;
    const uint32_t bar0 = smem_u32(bars);
    const uint32_t acc_full = bar0 + 16u * S, acc_empty = acc_full + 16u, w_full = acc_empty + 16u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t acc_cols = (uint32_t)(p.zp * N);
    const uint32_t ncols = tmem_cols(2 * (int)acc_cols);
    const uint32_t blk = N * 16u;                       // one tap and chunk plane of the weights

    if (threadIdx.x == 0) {
        for (int s = 0; s < 2 * S; ++s) mbar_init(bar0 + 8u * s, 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(acc_full + 8u * b, 1);
            mbar_init(acc_empty + 8u * b, kSlabEpiWarps);
        }
        mbar_init(w_full, 1);
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(tmem_slot), ncols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // weights: [dx][kc][dy][j][n][8] with j = 1 - dz, the order of the
        // output planes z - 1, z, z + 1 (the packed operand has [dz][dy])
        if (lane == 0) mbar_expect_tx(w_full, p.w_bytes);
        __syncwarp();
        const int nblk = 27 * p.kc_total;
        for (int i = lane; i < nblk; i += 32) {
            const int t9 = i % 9, dz = t9 / 3, dy = t9 % 3;
            bulk_load(wbase + (uint32_t)(i - t9 + 3 * dy + 2 - dz) * blk,
                      p.wpack + (size_t)i * (N * 8), blk, w_full);
        }
        if (lane == 0) {
            Ring q;
            bool ok = true;
            for (int t = blockIdx.x; ok && t < p.tiles; t += gridDim.x) {
                int x0, y0, z0, b0;
                tile_origin_u32(p.g, (uint32_t)t, x0, y0, z0, b0);
                for (int dx = -1; ok && dx <= 1; ++dx)
                    for (int kc = 0; ok && kc < p.kc_total; kc += 2) {
                        const int mi = kc < p.kc0 ? 0 : 1, c8 = kc < p.kc0 ? kc : kc - p.kc0;
                        for (int z = 0; z < ZST; ++z, q.next(S)) {
                            const uint32_t full = bar0 + 8u * q.s, empty = bar0 + 8u * (S + q.s);
                            if (q.r > 0 && !mbar_wait(empty, (q.r - 1) & 1u, kWaitLimitNs)) {
                                atomicOr(p.err, ERR_TIMEOUT);
                                ok = false;
                                break;
                            }
                            mbar_expect_tx(full, p.stage_bytes);
                            tma_load_5d(sbase + (uint32_t)q.s * p.stage_bytes, &p.maps[mi], full, 8 * (x0 + dx),
                                        y0 - 1, z0 - 1 + z * ZC, b0, c8);
                        }
                    }
            }
        }
    } else if (warp == 1) {
        slab_issue<N, ZC, ZST>(p, bar0, acc_full, acc_empty, w_full, wbase, sbase, tmem);
    } else {
        const int q = warp & 3;
        const int r = q * 32 + lane;
        const int half = (warp - 2) >> 2;
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        const long long zstep = (long long)p.g.H * p.g.W;
        // ReLU masks of a plane, loaded a plane (the first: an accumulator wait)
        // ahead (64^3 32 -> 32, batch 16: 199 us; 228 where each chunk waits for its own)
        auto load_masks = [&](long long vox, uint4 (&mk)[N / 8]) {
#pragma unroll
            for (int n0 = 0; n0 < N; n0 += 16) {
                const EpiDest& d = (n0 < p.split) ? p.d[0] : p.d[1];
                if (d.mask == nullptr || d.out == nullptr) continue;
                const __nv_bfloat16* src = d.mask + ((n0 - d.col0) >> 3) * d.plane + vox * 8;
                mk[n0 / 8] = *reinterpret_cast<const uint4*>(src);
                mk[n0 / 8 + 1] = *reinterpret_cast<const uint4*>(src + d.plane);
            }
        };
        const bool masks = p.d[0].mask != nullptr || p.d[1].mask != nullptr;
        uint32_t it = 0;
        for (int t = blockIdx.x; t < p.tiles; t += gridDim.x, ++it) {
            const uint32_t buf = it & 1u, use = it >> 1;
            int x0, y0, z0, b0;
            tile_origin_u32(p.g, (uint32_t)t, x0, y0, z0, b0);
            const int x = x0 + r % p.g.bx, y = y0 + r / p.g.bx;
            // two warps per quarter of the rows: even and odd planes
            long long vox = (((long long)b0 * p.g.D + z0 + half) * p.g.H + y) * p.g.W + x;
            uint4 mk[N / 8], next[N / 8];
            if (masks) load_masks(vox, next);
            if (!__all_sync(0xffffffffu, mbar_wait(acc_full + 8u * buf, use & 1u, kWaitLimitNs))) {
                if (lane == 0) atomicOr(p.err, ERR_TIMEOUT);
                break;
            }
            tc_fence_after();
            for (int z = half; z < p.zp; z += 2, vox += 2 * zstep) {
                const uint32_t col = tmem + buf * acc_cols + lane_base + (uint32_t)(z * N);
                float head = 0.f;
                if (masks) {
#pragma unroll
                    for (int i = 0; i < N / 8; ++i) mk[i] = next[i];
                    if (z + 2 < p.zp) load_masks(vox + 2 * zstep, next);
                }
#pragma unroll
                for (int n0 = 0; n0 < N; n0 += 16) {
                    uint32_t v[16];
                    tmem_ld16(col + (uint32_t)n0, v);
                    tmem_wait_ld();
                    const EpiDest& d = (n0 < p.split) ? p.d[0] : p.d[1];
                    if (d.out == nullptr) continue;
                    const int ch0 = n0 - d.col0;
                    emit16(d, v, ch0, (ch0 >> 3) * d.plane + vox * 8, p.head_out ? p.head_w : nullptr, head,
                           &mk[n0 / 8]);
                }
                if (p.head_out) p.head_out[vox] = head + *p.head_b;
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty + 8u * buf);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, ncols);
    }
}

template <int N, int ZC, int ZST>
cudaError_t launch_slab_as(const SlabParams& p, int grid, size_t smem, cudaStream_t s) {
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(slab_kernel<N, ZC, ZST>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             227 * 1024);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    slab_kernel<N, ZC, ZST><<<grid, kSlabThreads, smem, s>>>(p);
    return cudaGetLastError();
}

template <int N>
cudaError_t launch_slab_n(const SlabParams& p, int grid, size_t smem, cudaStream_t s) {
    switch (p.zp) {                 // stages as in slab_zc
    case 2: return launch_slab_as<N, 2, 2>(p, grid, smem, s);
    case 4: return launch_slab_as<N, 3, 2>(p, grid, smem, s);
    case 8: if (N <= 32) return launch_slab_as<N <= 32 ? N : 16, 5, 2>(p, grid, smem, s); break;
    case 16: if (N <= 16) return launch_slab_as<16, 6, 3>(p, grid, smem, s); break;
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_slab(const SlabParams& p, int grid, size_t smem, cudaStream_t s) {
    switch (p.n) {
    case 16: return launch_slab_n<16>(p, grid, smem, s);
    case 32: return launch_slab_n<32>(p, grid, smem, s);
    case 64: return launch_slab_n<64>(p, grid, smem, s);
    }
    return cudaErrorInvalidValue;
}

__global__ void __launch_bounds__(kThreads, 1) rows_kernel(const __grid_constant__ RowsParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    const int S = p.stages;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)S * p.stage_bytes);
    volatile int* tile_slot = reinterpret_cast<volatile int*>(bars + 2 * S + 12);   // [4]
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S + 14);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bar0 = smem_u32(bars);
    const uint32_t acc_full = bar0 + 16u * S, acc_empty = acc_full + 16u;   // [2] each
    const uint32_t tile_full = acc_empty + 16u, tile_empty = tile_full + 32u;   // [4] each
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t acc_cols = (uint32_t)(p.mt * p.n_tile);   // one accumulator per subtile
    const uint32_t ncols = tmem_cols(p.nbuf * (int)acc_cols);

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(bar0 + 8u * s, 1);
            mbar_init(bar0 + 8u * (S + s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(acc_full + 8u * b, 1);
            mbar_init(acc_empty + 8u * b, 4);
        }
        for (int b = 0; b < 4; ++b) {
            mbar_init(tile_full + 8u * b, 1);
            mbar_init(tile_empty + 8u * b, 5);   // the MMA warp and the four epilogue warps
        }
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(tmem_slot), ncols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    int* const tile_ctr = p.tile_ctr + blockIdx.y;

    const bool conv = p.tap_mode == TAP_SHIFT3;
    if (warp == 0) {
        if (lane == 0) {
            const int gpt = conv ? p.kc_total / p.E : p.kc_total / p.kc_step;
            const uint32_t tx = p.a_stage_bytes + p.b_stage_bytes;
            Ring q;
            bool ok = true;
            int claimed = atomicAdd(tile_ctr, 1);
            for (uint32_t it = 0; ok; ++it) {
                // publish the claimed tile's index (-1: none left) in slot it % 4
                const uint32_t ts = it & 3u, tu = it >> 2;
                if (tu > 0 && !mbar_wait(tile_empty + 8u * ts, (tu - 1) & 1u, kWaitLimitNs)) {
                    atomicOr(p.err, ERR_TIMEOUT);
                    break;
                }
                const int t = claimed < p.tiles ? claimed : -1;
                tile_slot[ts] = t;
                mbar_arrive(tile_full + 8u * ts);
                if (t < 0) break;
                // claim the following tile now: the atomic's latency hides behind this tile's loads
                claimed = atomicAdd(tile_ctr, 1);
                int x0, y0, z0, b0;
                tile_origin_u32(p.g, (uint32_t)t, x0, y0, z0, b0);
                int tap = 0, g = 0;   // K-step k = tap * gpt + g
                for (int k = 0; k < p.ksteps; ++k, q.next(S), g = (g + 1 < gpt) ? g + 1 : 0, tap += (g == 0)) {
                    const int s = q.s;
                    const uint32_t r = q.r;
                    const uint32_t full = bar0 + 8u * s, empty = bar0 + 8u * (S + s);
                    if (r > 0 && !mbar_wait(empty, (r - 1) & 1u, kWaitLimitNs)) {
                        atomicOr(p.err, ERR_TIMEOUT);
                        ok = false;
                        break;
                    }
                    mbar_expect_tx(full, tx);
                    const uint32_t a_dst = sbase + (uint32_t)s * p.stage_bytes;
                    if (conv && p.halo == 2) {
                        // full halo: one box of (bx + 2, by + 2, 3) voxels per block of E planes
                        // holds all 27 taps; the weights of the three x-shifts follow
                        const int kc = k * p.E;
                        const int mi = kc < p.kc0 ? 0 : 1, c8 = kc < p.kc0 ? kc : kc - p.kc0;
                        tma_load_5d(a_dst, &p.maps[mi], full, 8 * (x0 - 1), y0 - 1, z0 - 1, b0, c8);
                        const uint32_t bsz = 9u * p.E * p.n_tile * 16u;
                        for (int dxi = 0; dxi < 3; ++dxi) {
                            const __nv_bfloat16* src =
                                p.wpack + ((size_t)(blockIdx.y * 3 + dxi) * p.kc_total + kc) * 9 * p.n_tile * 8;
                            bulk_load(a_dst + p.a_stage_bytes + bsz * dxi, src, bsz, full);
                        }
                    } else if (conv) {
                        // tap = x-shift index, g = block of E chunk planes
                        const int dx = tap - 1, kc = g * p.E;
                        const int mi = kc < p.kc0 ? 0 : 1, c8 = kc < p.kc0 ? kc : kc - p.kc0;
                        if (p.halo) {
                            tma_load_5d(a_dst, &p.maps[mi], full, 8 * (x0 + dx), y0 - 1, z0 - 1, b0, c8);
                        } else {
                            for (int t9 = 0; t9 < 9; ++t9)
                                tma_load_5d(a_dst + (uint32_t)(t9 * p.E) * 2048u, &p.maps[mi], full, 8 * (x0 + dx),
                                            y0 + (t9 % 3) - 1, z0 + (t9 / 3) - 1, b0, c8);
                        }
                        const __nv_bfloat16* src =
                            p.wpack + ((size_t)(blockIdx.y * 3 + tap) * p.kc_total + kc) * 9 * p.n_tile * 8;
                        bulk_load(a_dst + p.a_stage_bytes, src, p.b_stage_bytes, full);
                    } else {
                        if (p.tap_mode == TAP_MAP) {
                            for (int j = 0; j < p.kc_step; ++j)
                                load_box(a_dst + 2048u * j, &p.maps[tap], full, true, g * p.kc_step + j, x0, y0, z0,
                                         b0, p.g.B);
                        } else {
                            // TAP_NONE: one box of kc_step chunk planes
                            tma_load_5d(a_dst, &p.maps[0], full, 8 * x0, y0, z0, b0, g * p.kc_step);
                        }
                        const __nv_bfloat16* src =
                            p.wpack + ((size_t)(blockIdx.y * p.n_taps + tap) * p.kc_total + (size_t)g * p.kc_step) *
                                          p.n_tile * 8;
                        bulk_load(a_dst + p.a_stage_bytes, src, p.b_stage_bytes, full);
                    }
                }
            }
        }
    } else if (warp == 1) {
        // The whole warp walks the K-steps, so the descriptor arithmetic stays
        // warp-uniform; one elected lane issues every MMA and commit.
        const bool leader = elect_one();
        const uint32_t nrow = (uint32_t)p.n_tile * 16u;   // bytes of one packed chunk of B
        // conv3 with halo 0 / 1: start offsets (16-byte units) of the nine (dz, dy)
        // taps and the A operand's K-direction core-matrix stride
        const uint32_t a_lbo = p.halo == 1 ? p.halo_plane : 2048u;
        uint32_t tap_off[9];
#pragma unroll
        for (int t9 = 0; t9 < 9; ++t9)
            tap_off[t9] = p.halo == 1 ? (uint32_t)(((t9 / 3) * (p.g.by + 2) + (t9 % 3)) * p.g.bx)
                                      : (uint32_t)(t9 * p.E) * 128u;
        Ring q;
        bool ok = true;
        for (uint32_t it = 0; ok; ++it) {
            const uint32_t ts = it & 3u, tu = it >> 2;
            if (!__all_sync(0xffffffffu, mbar_wait(tile_full + 8u * ts, tu & 1u, kWaitLimitNs))) {
                if (leader) atomicOr(p.err, ERR_TIMEOUT);
                break;
            }
            const int t = tile_slot[ts];
            __syncwarp();
            if (leader) mbar_arrive(tile_empty + 8u * ts);
            if (t < 0) break;
            // accumulator buffer of this tile and how often it was filled before
            const uint32_t buf = p.nbuf == 2 ? (it & 1u) : 0u, use = p.nbuf == 2 ? (it >> 1) : it;
            if (use > 0 && !__all_sync(0xffffffffu, mbar_wait(acc_empty + 8u * buf, (use - 1) & 1u, kWaitLimitNs))) {
                if (leader) atomicOr(p.err, ERR_TIMEOUT);
                break;
            }
            tc_fence_after();
            const uint32_t acc = tmem + buf * acc_cols;
            for (int k = 0; k < p.ksteps; ++k, q.next(S)) {
                const int s = q.s;
                const uint32_t r = q.r;
                if (!__all_sync(0xffffffffu, mbar_wait(bar0 + 8u * s, r & 1u, kWaitLimitNs))) {
                    if (leader) atomicOr(p.err, ERR_TIMEOUT);
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t a0 = sbase + (uint32_t)s * p.stage_bytes;
                const uint32_t b0s = a0 + p.a_stage_bytes;
                if (conv && p.halo == 2) {
                    if (leader) {
                        // rows of a subtile are y-runs of bx = 8 voxels: one core-matrix group
                        // each, (bx + 2) * 16 bytes apart in the halo box; every tap is a
                        // start offset ((dz, dy) rows, dx * 16 bytes)
                        const uint32_t rowb = (uint32_t)(p.g.bx + 2) * 16u;
                        const uint32_t sub = (uint32_t)(kRows / p.g.bx) * rowb;
                        const uint32_t bsz = 9u * p.E * nrow;
                        for (int dxi = 0; dxi < 3; ++dxi)
                            for (int t9 = 0; t9 < 9; ++t9) {
                                const uint32_t a_tap =
                                    a0 + (uint32_t)((t9 / 3) * (p.g.by + 2) + (t9 % 3)) * rowb + 16u * dxi;
                                for (int i = 0; i < p.E / 2; ++i) {
                                    const uint64_t bd =
                                        smem_desc(b0s + bsz * dxi + (uint32_t)(2 * i * 9 + t9) * nrow, 9u * nrow, 128);
                                    for (int m = 0; m < p.mt; ++m) {
                                        const uint64_t ad =
                                            smem_desc(a_tap + sub * m + 2u * i * p.halo_plane, p.halo_plane, rowb);
                                        umma_bf16(acc + (uint32_t)(m * p.n_tile), ad, bd, p.idesc,
                                                  (k > 0 || dxi > 0 || t9 > 0 || i > 0) ? 1u : 0u);
                                    }
                                }
                            }
                    }
                } else if (conv) {
                    const uint64_t ad = smem_desc(a0, a_lbo, 128), bd = smem_desc(b0s, 9u * nrow, 128);
                    if (leader)
                        issue_conv_step(p.mt, p.E / 2, acc, ad, bd, tap_off, a_lbo / 8u, (uint32_t)p.n_tile, p.idesc,
                                        k == 0);
                } else if (leader) {
                    for (int i = 0; i < p.kc_step / 2; ++i) {
                        const uint64_t ad = smem_desc(a0 + 4096u * i, 2048u, 128);
                        const uint64_t bd = smem_desc(b0s + 2u * i * nrow, nrow, 128);
                        umma_bf16(acc, ad, bd, p.idesc, (k > 0 || i > 0) ? 1u : 0u);
                    }
                }
                if (leader) umma_commit(bar0 + 8u * (S + s));
                __syncwarp();
            }
            if (!ok) break;
            if (leader) umma_commit(acc_full + 8u * buf);
            __syncwarp();
        }
    } else {
        const int q = warp & 3;
        const int r = q * 32 + lane;
        for (uint32_t it = 0;; ++it) {
            const uint32_t ts = it & 3u, tu = it >> 2;
            if (!__all_sync(0xffffffffu, mbar_wait(tile_full + 8u * ts, tu & 1u, kWaitLimitNs))) {
                if (lane == 0) atomicOr(p.err, ERR_TIMEOUT);
                break;
            }
            const int t = tile_slot[ts];
            __syncwarp();
            if (lane == 0) mbar_arrive(tile_empty + 8u * ts);
            if (t < 0) break;
            const uint32_t buf = p.nbuf == 2 ? (it & 1u) : 0u, use = p.nbuf == 2 ? (it >> 1) : it;
            if (!__all_sync(0xffffffffu, mbar_wait(acc_full + 8u * buf, use & 1u, kWaitLimitNs))) {
                if (lane == 0) atomicOr(p.err, ERR_TIMEOUT);
                break;
            }
            {
                tc_fence_after();
                const uint32_t acc = tmem + buf * acc_cols;
                int x0, y0, z0, b0;
                tile_origin_u32(p.g, (uint32_t)t, x0, y0, z0, b0);
                const uint32_t lane_base = (uint32_t)(q * 32) << 16;
                const int nch = p.n_tile / 16;
                // up layers: column n = o n_up + channel, o = (oz, oy, ox) the fine offset
                const long long fW = 2LL * p.g.W, fHW = fW * (2LL * p.g.H);
                for (int m = 0; m < p.mt; ++m) {
                    int vx, vy, vz, vb;
                    const long long vox = row_voxel(p.g, x0, y0, z0, b0, m * kRows + r, &vx, &vy, &vz, &vb);
                    // fine voxel (2 vx, 2 vy, 2 vz) of sample vb (up layers)
                    const long long fine0 = ((long long)vb * (2 * p.g.D) + 2 * vz) * fHW + 2LL * vy * fW + 2 * vx;
                    float head_acc = 0.f;
                    // epilogue of accumulator chunk j (16 columns)
                    auto emit = [&](int j, const uint32_t (&v)[16]) {
                        const int n0 = blockIdx.y * p.n_tile + j * 16;
                        const EpiDest& d = (n0 < p.split) ? p.d[0] : p.d[1];
                        if (d.out == nullptr) return;
                        int ch0;
                        long long off;
                        if (p.scatter_up) {
                            const int o = n0 / p.cout_up;
                            ch0 = n0 - o * p.cout_up;
                            const long long fine = fine0 + (o >> 2) * fHW + ((o >> 1) & 1) * fW + (o & 1);
                            off = (ch0 >> 3) * d.plane + fine * 8;
                        } else {
                            ch0 = n0 - d.col0;
                            off = (ch0 >> 3) * d.plane + vox * 8;
                        }
                        emit16(d, v, ch0, off, p.head_out ? p.head_w : nullptr, head_acc);
                    };
                    for (int j = 0; j < nch; ++j) {
                        uint32_t v[16];
                        tmem_ld16(acc + lane_base + (uint32_t)(m * p.n_tile + j * 16), v);
                        tmem_wait_ld();
                        emit(j, v);
                    }
                    if (p.head_out) p.head_out[vox] = head_acc + *p.head_b;
                }
            }
            // this warp's reads of the buffer are complete: hand it back to the MMA warp
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty + 8u * buf);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, ncols);
    }
}

// ------------------------------------------------------------------------
// Weight-gradient GEMM.  Per K-step (64 voxels of the V grid) the producer
// loads, for each of the tile's 16 row groups, a 64 x 16-byte box of the
// group's (tap, 8-channel chunk) input view, and the n/8 boxes of the output
// gradient: both operands are MN-major (8 channels contiguous per voxel).
// A row group may be the bias group: constant ones, so its rows accumulate
// sum_v dY[v, n], the bias gradient.
// ------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads, 1) wgrad_kernel(const __grid_constant__ WgradParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    const int S = p.stages;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)S * p.stage_bytes);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S + 1);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bar0 = smem_u32(bars);
    const uint32_t done = bar0 + 16u * S;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t ncols = tmem_cols(p.n);
    const int g0 = blockIdx.y * 16;
    const int groups_all = p.n_groups + (p.ones_group >= 0 ? 1 : 0);
    const int ng = min(16, groups_all - g0);
    const int btap = blockIdx.z;
    const int kbeg = blockIdx.x * p.ksteps_per_cta;
    const int kend = min(kbeg + p.ksteps_per_cta, p.ksteps_total);

    const uint32_t gbytes = (uint32_t)p.kv * 16u;   // one group's block of a stage
    // bias group: bf16 ones in its slot of every stage (written once, never loaded over)
    const int ones_slot = (p.ones_group >= g0 && p.ones_group < g0 + 16) ? p.ones_group - g0 : -1;
    if (ones_slot >= 0) {
        for (int s = 0; s < S; ++s) {
            uint32_t* dst = reinterpret_cast<uint32_t*>(smem + (size_t)s * p.stage_bytes + gbytes * ones_slot);
            for (int i = threadIdx.x; i < (int)(gbytes / 4); i += blockDim.x) dst[i] = 0x3F803F80u;
        }
        fence_async_shared();
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(bar0 + 8u * s, 1);
            mbar_init(bar0 + 8u * (S + s), 1);
        }
        mbar_init(done, 1);
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(tmem_slot), ncols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // the whole warp walks the K-steps; one elected lane issues (see rows_kernel)
        const bool leader = elect_one();
        int real = 0;
        for (int sl = 0; sl < ng; ++sl) real += (sl != ones_slot);
        const uint32_t tx = gbytes * real + (uint32_t)(p.n / 8) * gbytes;
        // every K-step loads the same slots: lane sl decodes slot sl once (source
        // map mi, chunk plane c8, tap shift), packed mi | c8 << 4 | (dx, dy, dz) + 1
        // in bits 14, 16, 18
        int code = 0;
        if (lane < ng && lane != ones_slot) {
            const int g = g0 + lane;
            int mi = 0, c8, dx = 0, dy = 0, dz = 0;
            if (p.mode == KIND_CONV3) {
                const int tap = g / p.kc_total;
                c8 = g % p.kc_total;
                dz = tap / 9 - 1;
                dy = (tap / 3) % 3 - 1;
                dx = tap % 3 - 1;
                if (c8 >= p.kc0) {
                    mi = 1;
                    c8 -= p.kc0;
                }
            } else if (p.mode == KIND_DOWN) {
                mi = g / p.kc_total;
                c8 = g % p.kc_total;
            } else {
                c8 = g;
            }
            code = mi | (c8 << 4) | ((dx + 1) << 14) | ((dy + 1) << 16) | ((dz + 1) << 18);
        }
        Ring q;
        int x0, y0, z0, b0;
        tile_origin(p.g, kbeg, x0, y0, z0, b0);
        for (int k = kbeg; k < kend; ++k, q.next(S), tile_next(p.g, x0, y0, z0, b0)) {
            const int kk = k - kbeg;
            const int s = q.s;
            const uint32_t r = q.r;
            const uint32_t full = bar0 + 8u * s, empty = bar0 + 8u * (S + s);
            if (kk >= S && !__all_sync(0xffffffffu, mbar_wait(empty, (r - 1) & 1u, kWaitLimitNs))) {
                if (leader) atomicOr(p.err, ERR_TIMEOUT);
                break;
            }
            if (leader) mbar_expect_tx(full, tx);
            const uint32_t a_dst = sbase + (uint32_t)s * p.stage_bytes;
            for (int sl = 0; sl < ng;) {
                if (sl == ones_slot) {
                    ++sl;
                    continue;
                }
                const int c = __shfl_sync(0xffffffffu, code, sl);
                const int mi = c & 15, c8 = (c >> 4) & 1023;
                const int dx = ((c >> 14) & 3) - 1, dy = ((c >> 16) & 3) - 1, dz = ((c >> 18) & 3) - 1;
                // one box brings ea consecutive chunk planes (runs never straddle a tap or source)
                if (leader)
                    load_box(a_dst + gbytes * sl, &p.amaps[mi], full, p.mode == KIND_DOWN, c8, x0 + dx, y0 + dy,
                             z0 + dz, b0, p.g.B);
                sl += p.ea;
            }
            const CUtensorMap* bm = &p.bmaps[p.mode == KIND_UP ? btap : 0];
            for (int j = 0; j < p.n / 8; j += p.eb)
                if (leader)
                    load_box(a_dst + p.a_stage_bytes + gbytes * j, bm, full, p.mode == KIND_UP, j, x0, y0, z0, b0,
                             p.g.B);
            __syncwarp();
        }
    } else if (warp == 1) {
        // the whole warp walks the K-steps; one elected lane issues (see rows_kernel)
        const bool leader = elect_one();
        Ring q;
        for (int k = kbeg; k < kend; ++k, q.next(S)) {
            const int kk = k - kbeg;
            const int s = q.s;
            const uint32_t r = q.r;
            if (!__all_sync(0xffffffffu, mbar_wait(bar0 + 8u * s, r & 1u, kWaitLimitNs))) {
                if (leader) atomicOr(p.err, ERR_TIMEOUT);
                break;
            }
            tc_fence_after();
            const uint32_t a0 = sbase + (uint32_t)s * p.stage_bytes;
            const uint32_t b0s = a0 + p.a_stage_bytes;
            // K-slice i starts 256 bytes (16 units) further in both operands
            const uint64_t ad = smem_desc(a0, 128u, gbytes), bd = smem_desc(b0s, 128u, gbytes);
            if (leader) {
                for (int i = 0; i < p.kv / 16; ++i)
                    umma_bf16(tmem, ad + 16u * i, bd + 16u * i, p.idesc, (kk > 0 || i > 0) ? 1u : 0u);
                umma_commit(bar0 + 8u * (S + s));
            }
            __syncwarp();
        }
        if (leader) umma_commit(done);
        __syncwarp();
    } else {
        const int q = warp & 3;
        const int r = q * 32 + lane;
        const int sl = r >> 3, r8 = r & 7;
        const int g = g0 + sl;
        bool ok = mbar_wait(done, 0, kWaitLimitNs);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) {
            if (lane == 0) atomicOr(p.err, ERR_TIMEOUT);
        } else if (kend > kbeg) {
            tc_fence_after();
            float* dst = nullptr;
            if (sl < ng) {
                if (g == p.ones_group) {
                    dst = (r8 == 0) ? p.db : nullptr;
                } else {
                    int tap, c8;
                    if (p.mode == KIND_UP) {
                        tap = btap;
                        c8 = g;
                    } else {
                        tap = g / p.kc_total;
                        c8 = g % p.kc_total;
                    }
                    dst = p.dw + ((size_t)(tap * p.kc_total + c8) * 8 + r8) * p.n;
                }
            }
            for (int j = 0; j < p.n / 16; ++j) {
                uint32_t v[16];
                tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(j * 16), v);
                tmem_wait_ld();
                if (dst) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) atomicAdd(dst + j * 16 + i, __uint_as_float(v[i]));
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, ncols);
    }
}

cudaError_t launch_rows(const RowsParams& p, int grid_n, size_t smem, cudaStream_t s) {
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(rows_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                     cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    // resident CTAs per SM: the occupancy query's answer, at most 512 / ncols
    // by TMEM (a CTA beyond that would wait in tcgen05.alloc for a whole
    // persistent CTA).  The grid is `persistent` times that many CTAs per SM:
    // tiles are claimed dynamically, so a surplus CTA finds none and exits.
    int dev = 0, sms = 0, occ = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, rows_kernel, kThreads, smem);
    if (e != cudaSuccess) return e;
    const int by_tmem = 512 / (int)tmem_cols(p.nbuf * p.mt * p.n_tile);
    const int per_sm = occ < by_tmem ? occ : by_tmem;
    long long grid_m = (long long)sms * (per_sm > 0 ? per_sm : 1) * (p.persistent > 0 ? p.persistent : 1);
    if (grid_m > p.tiles || !p.persistent) grid_m = p.tiles;
    rows_kernel<<<dim3((unsigned)grid_m, grid_n), kThreads, smem, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_wgrad(const WgradParams& p, dim3 grid, size_t smem, cudaStream_t s) {
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    wgrad_kernel<<<grid, kThreads, smem, s>>>(p);
    return cudaGetLastError();
}

}  // namespace spnn

namespace spnn {

// K-step walk of the halo weight gradient: x-runs of rl voxels fastest, then z
// within a slab of zs planes, then y, then the slab, then the sample, so that
// the (dz, dy) halo rows a K-step loads were loaded by a recent K-step (L2).
struct HaloWalk {
    int xr, zi, y, zsl, b;
    __device__ __forceinline__ void start(const WgradHaloParams& p, int k) {
        xr = k % p.nx;
        k /= p.nx;
        zi = k % p.zs;
        k /= p.zs;
        y = k % p.g.H;
        k /= p.g.H;
        zsl = k % p.nzs;
        b = k / p.nzs;
    }
    __device__ __forceinline__ void next(const WgradHaloParams& p) {
        if (++xr < p.nx) return;
        xr = 0;
        if (++zi < p.zs) return;
        zi = 0;
        if (++y < p.g.H) return;
        y = 0;
        if (++zsl < p.nzs) return;
        zsl = 0;
        ++b;
    }
    __device__ __forceinline__ int x0(const WgradHaloParams& p) const { return p.rl * xr; }
    __device__ __forceinline__ int z0(const WgradHaloParams& p) const { return zsl * p.zs + zi; }
};

__global__ void __launch_bounds__(kThreads, 1) wgrad_halo_kernel(const __grid_constant__ WgradHaloParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    const int S = p.stages;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)S * p.stage_bytes);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S + 1);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bar0 = smem_u32(bars);
    const uint32_t done = bar0 + 16u * S;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int kbeg = blockIdx.x * p.ksteps_per_cta;
    const int kend = min(kbeg + p.ksteps_per_cta, p.ksteps_total);
    // this CTA's planes: npc planes of one source from plane `first` on (planes
    // past the source's end load as zeros), `real` of them inside the source
    const int split = blockIdx.y;
    const int src = split < p.splits0 ? 0 : 1;
    const int npc = src ? p.npc1 : p.npc0;
    const int first = (src ? split - p.splits0 : split) * npc;
    const int real = min(npc, (src ? p.kc1 : p.kc0) - first);
    const int plane_off = (src ? p.kc0 : 0) + first;       // in the concatenated input
    const int groups = 9 * npc;                            // row group `groups` is the ones row
    const int nM = (groups + 16) / 16;                     // 128-row tiles holding groups + 1
    const uint32_t n3 = 3u * (uint32_t)p.n;                 // MMA N: (dx, output channel)
    const uint32_t ncols = tmem_cols(nM * (int)n3);
    const uint32_t row = 16u * (uint32_t)p.rl;             // bytes of one run of one chunk plane

    // the ones row of every K-step region of every stage (written once; TMA never writes it)
    for (int s = 0; s < S * p.ksub; ++s) {
        uint32_t* dst = reinterpret_cast<uint32_t*>(smem + (size_t)(s / p.ksub) * p.stage_bytes +
                                                    (size_t)(s % p.ksub) * p.sub_bytes + (size_t)groups * row);
        for (int i = threadIdx.x; i < (int)(row / 4); i += blockDim.x) dst[i] = 0x3F803F80u;
    }
    fence_async_shared();
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(bar0 + 8u * s, 1);
            mbar_init(bar0 + 8u * (S + s), 1);
        }
        mbar_init(done, 1);
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(tmem_slot), ncols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // the whole warp walks the K-steps; one elected lane issues (see rows_kernel)
        const bool leader = elect_one();
        const uint32_t b_box = (uint32_t)(p.n / 8) * row;   // n/8 planes of one run
        const uint32_t tx = (uint32_t)groups * row + 3u * b_box;
        Ring q;
        HaloWalk w;
        w.start(p, kbeg);
        // a stage holds ns <= ksub consecutive K-steps
        for (int k = kbeg; k < kend; q.next(S)) {
            const int ns = min(p.ksub, kend - k);
            const int s = q.s;
            const uint32_t r = q.r;
            const uint32_t full = bar0 + 8u * s, empty = bar0 + 8u * (S + s);
            if (r > 0 && !__all_sync(0xffffffffu, mbar_wait(empty, (r - 1) & 1u, kWaitLimitNs))) {
                if (leader) atomicOr(p.err, ERR_TIMEOUT);
                break;
            }
            if (leader) mbar_expect_tx(full, (uint32_t)ns * tx);
            for (int j = 0; j < ns; ++j, w.next(p)) {
                const uint32_t a_dst = sbase + (uint32_t)s * p.stage_bytes + (uint32_t)j * p.sub_bytes;
                if (leader) {
                    const int x0 = w.x0(p), z0 = w.z0(p);
                    // input: (rl, 3, 3) voxels of npc planes, rows (plane, dz, dy)
                    tma_load_5d(a_dst, &p.amaps[src], full, 8 * x0, w.y - 1, z0 - 1, w.b, first);
                    // output gradient shifted by -dx: B block dxi holds dY at x - (dxi - 1)
                    for (int dxi = 0; dxi < 3; ++dxi)
                        tma_load_5d(a_dst + p.a_region + (uint32_t)dxi * b_box, &p.bmap, full, 8 * (x0 + 1 - dxi),
                                    w.y, z0, w.b, 0);
                }
            }
            k += ns;
            __syncwarp();
        }
    } else if (warp == 1) {
        // the whole warp walks the K-steps; one elected lane issues (see rows_kernel)
        const bool leader = elect_one();
        Ring q;
        for (int k = kbeg; k < kend; q.next(S)) {
            const int ns = min(p.ksub, kend - k);
            const int s = q.s;
            const uint32_t r = q.r;
            if (!__all_sync(0xffffffffu, mbar_wait(bar0 + 8u * s, r & 1u, kWaitLimitNs))) {
                if (leader) atomicOr(p.err, ERR_TIMEOUT);
                break;
            }
            tc_fence_after();
            for (int j = 0; j < ns; ++j) {
                const uint32_t a0 = sbase + (uint32_t)s * p.stage_bytes + (uint32_t)j * p.sub_bytes;
                // MN-major operands: 8-voxel core matrices 128 bytes apart along K,
                // 8-channel groups one run apart along M / N; K-block kb = voxels
                // 16 kb .. 16 kb + 15 of the run, a 256-byte start offset
                if (leader)
                    for (int kb = 0; kb < p.rl / 16; ++kb) {
                        const uint64_t bd = smem_desc(a0 + p.a_region + 256u * kb, 128u, row);
                        for (int m = 0; m < nM; ++m)
                            umma_bf16(tmem + (uint32_t)m * n3, smem_desc(a0 + (uint32_t)m * 16u * row + 256u * kb, 128u, row),
                                      bd, p.idesc, (k > kbeg || j > 0 || kb > 0) ? 1u : 0u);
                    }
            }
            if (leader) umma_commit(bar0 + 8u * (S + s));
            k += ns;
            __syncwarp();
        }
        if (leader) umma_commit(done);
        __syncwarp();
    } else {
        const int q = warp & 3;
        const int r = q * 32 + lane;
        bool ok = mbar_wait(done, 0, kWaitLimitNs);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) {
            if (lane == 0) atomicOr(p.err, ERR_TIMEOUT);
        } else if (kend > kbeg) {
            tc_fence_after();
            const int ci_all = 8 * (p.kc0 + p.kc1);
            for (int m = 0; m < nM; ++m) {
                const int g = 16 * m + (r >> 3), r8 = r & 7;
                const int pl = g / 9, t9 = g % 9;             // t9 = (dz + 1) * 3 + (dy + 1)
                const bool wrow = g < groups && pl < real;
                const bool orow = g == groups && r8 == 0 && split == p.ones_split;
                for (uint32_t c = 0; c < n3; c += 16) {
                    uint32_t v[16];
                    tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)m * n3 + c, v);
                    tmem_wait_ld();
                    const int dxi = (int)c / p.n, co = (int)c % p.n;
                    float* dst = nullptr;
                    if (wrow)
                        dst = p.dw + ((size_t)(t9 * 3 + dxi) * ci_all + (plane_off + pl) * 8 + r8) * p.n + co;
                    else if (orow && dxi == 1)
                        dst = p.db + co;
                    if (dst) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) atomicAdd(dst + e, __uint_as_float(v[e]));
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, ncols);
    }
}

cudaError_t launch_wgrad_halo(const WgradHaloParams& p, dim3 grid, size_t smem, cudaStream_t s) {
    static bool attr = false;
    if (!attr) {
        cudaError_t e =
            cudaFuncSetAttribute(wgrad_halo_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    wgrad_halo_kernel<<<grid, kThreads, smem, s>>>(p);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------
// conv3 weight gradient on row windows (see WgradRowsParams).  N3 = 3 nc MMA
// columns, NM 128-row tiles (9 np groups of 8 rows, the rest reads what follows
// and is dropped), RPS output rows (pairs of rows where bx = 8) per K-step with
// KPR 16-voxel K-blocks each.
//
// What bounded the kernels before it was operand delivery: the halo kernel
// loaded nine input rows per plane for every output row and the per-tap kernel
// up to 16 boxes per K-step (tensor pipe 17 - 25 % active).  Here an input row
// is loaded (by + 2) / by times per z-plane, and a K-step is 8 to 24 MMAs issued
// as straight code.  Measured at batch 16, halo or per-tap kernel -> this: 64^3
// 16 -> 32 channels 272 -> 138 us, 32 -> 32 450 -> 200 us, 64 -> 32 801 -> 375 us
// (1.24 PFLOP/s); 32^3 64 -> 64 218 -> 117 us, 128 -> 64 412 -> 206 us; 16^3
// 128 -> 128 115 -> 78 us; 8^3 256 -> 256 128 -> 73 us.
// ------------------------------------------------------------------------

// The MMAs of one stage, straight line (a loop that works out its operands
// takes a lone warp longer than the MMAs).  Offsets in 16-byte units: a_row /
// b_row between output rows, 16 between K-blocks of a row, a_tile between M tiles.
template <int N3, int NM, int KPR, int RPS>
__device__ __forceinline__ void wgrad_rows_stage(uint32_t tmem, uint32_t a, uint32_t a_hi, uint32_t a_row,
                                                 uint32_t a_tile, uint32_t b, uint32_t b_hi, uint32_t b_row,
                                                 bool first) {
    constexpr uint32_t id = idesc_bf16(128, N3, 1, 1);
#pragma unroll
    for (int r = 0; r < RPS; ++r)
#pragma unroll
        for (int k = 0; k < KPR; ++k)
#pragma unroll
            for (int m = 0; m < NM; ++m) {
                const uint32_t ad = a + (uint32_t)r * a_row + 16u * k + (uint32_t)m * a_tile;
                const uint32_t bd = b + (uint32_t)r * b_row + 16u * k;
                if (r == 0 && k == 0 && first) umma_bf16_lo<0>(tmem + (uint32_t)(m * N3), ad, a_hi, bd, b_hi, id);
                else umma_bf16_lo<1>(tmem + (uint32_t)(m * N3), ad, a_hi, bd, b_hi, id);
            }
}

template <int N3, int NM, int KPR, int RPS>
__global__ void __launch_bounds__(kThreads, 1) wgrad_rows_kernel(const __grid_constant__ WgradRowsParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    const int S = p.stages;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)S * p.stage_bytes);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S + 1);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bar0 = smem_u32(bars);
    const uint32_t done = bar0 + 16u * S;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int kbeg = blockIdx.x * p.ksteps_per_cta;
    const int kend = min(kbeg + p.ksteps_per_cta, p.ksteps_total);
    constexpr int nb = N3 / 24;                            // 8-channel blocks of dY
    const int split = blockIdx.y, src = split < p.splits0 ? 0 : 1;
    const int np = src ? p.np1 : p.np0;
    const int first = (src ? split - p.splits0 : split) * np;      // planes past the source load as zeros
    const int real = min(np, (src ? p.kc1 : p.kc0) - first);
    const int co0 = blockIdx.z * p.nc;
    const bool bias = p.db != nullptr && split == 0;
    const uint32_t row = 16u * (uint32_t)p.bx;             // one x-run of 8 channels
    constexpr uint32_t ncols = (NM * N3 <= 64) ? 64 : (NM * N3 <= 128) ? 128 : (NM * N3 <= 256) ? 256 : 512;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(bar0 + 8u * s, 1);
            mbar_init(bar0 + 8u * (S + s), bias ? 5 : 1);  // the MMAs and, for the bias, four warps
        }
        mbar_init(done, 1);
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(tmem_slot), ncols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // lane 3 y + dx loads dY's row y shifted by dx, lane 31 the input box
        const int yl = lane / 3, dxl = lane % 3;
        const bool b_lane = lane < 3 * p.by;
        const uint32_t b_off = p.a_bytes + (uint32_t)lane * nb * row;
        const uint32_t tx = (uint32_t)(3 * np * (p.by + 2)) * row + (uint32_t)(3 * nb * p.by) * row;
        int k = kbeg, xr = k % p.nx, rest = k / p.nx;
        int zi = rest % p.zs;
        rest /= p.zs;
        int yb = rest % p.ny;
        rest /= p.ny;
        int zsl = rest % p.nzs, b = rest / p.nzs;
        Ring q;
        for (; k < kend; ++k, q.next(S)) {
            const uint32_t full = bar0 + 8u * q.s, empty = bar0 + 8u * (S + q.s);
            if (q.r > 0 && !__all_sync(0xffffffffu, mbar_wait(empty, (q.r - 1) & 1u, kWaitLimitNs))) {
                if (lane == 0) atomicOr(p.err, ERR_TIMEOUT);
                break;
            }
            if (lane == 0) mbar_expect_tx(full, tx);
            __syncwarp();
            const uint32_t dst = sbase + (uint32_t)q.s * p.stage_bytes;
            const int x0 = xr * p.bx, y0 = yb * p.by, z = zsl * p.zs + zi;
            if (b_lane) tma_load_5d(dst + b_off, &p.bmap, full, 8 * (x0 + 1 - dxl), co0 / 8, z, y0 + yl, b);
            if (lane == 31) tma_load_5d(dst, &p.amaps[src], full, 8 * x0, first, z - 1, y0 - 1, b);
            __syncwarp();
            // x-runs, then z within the slab, then y, slab, sample: the rows a
            // K-step loads were loaded by a recent one (L2)
            if (++xr == p.nx) {
                xr = 0;
                if (++zi == p.zs) {
                    zi = 0;
                    if (++yb == p.ny) {
                        yb = 0;
                        if (++zsl == p.nzs) zsl = 0, ++b;
                    }
                }
            }
        }
    } else if (warp == 1) {
        const bool leader = elect_one();
        // K-block of 16 voxels: two 8-voxel core matrices of one run, or (bx = 8)
        // of two rows; row groups one run apart
        const bool pairs = p.bx == 8;
        const uint32_t a_run = 3u * (uint32_t)np * row, b_run = 3u * nb * row;      // between output rows
        const uint64_t ad = smem_desc(sbase, pairs ? a_run : 128u, row);
        const uint64_t bd = smem_desc(sbase + p.a_bytes, pairs ? b_run : 128u, row);
        const uint32_t a_hi = (uint32_t)(ad >> 32), b_hi = (uint32_t)(bd >> 32), stage_u = p.stage_bytes / 16u;
        const uint32_t a_row = (pairs ? 2u : 1u) * a_run / 16u, b_row = (pairs ? 2u : 1u) * b_run / 16u;
        Ring q;
        for (int k = kbeg; k < kend; ++k, q.next(S)) {
            if (!__all_sync(0xffffffffu, mbar_wait(bar0 + 8u * q.s, q.r & 1u, kWaitLimitNs))) {
                if (leader) atomicOr(p.err, ERR_TIMEOUT);
                break;
            }
            tc_fence_after();
            if (leader) {
                wgrad_rows_stage<N3, NM, KPR, RPS>(tmem, (uint32_t)ad + (uint32_t)q.s * stage_u, a_hi, a_row, row,
                                                   (uint32_t)bd + (uint32_t)q.s * stage_u, b_hi, b_row, k == kbeg);
                umma_commit(bar0 + 8u * (S + q.s));
            }
            __syncwarp();
        }
        if (leader) umma_commit(done);
        __syncwarp();
    } else {
        const int q4 = warp & 3, r = q4 * 32 + lane;
        bool ok = true;
        if (bias) {
            // thread r sums channel block c8 of the voxels v = r % tpb + i tpb
            constexpr int tpb = 128 / nb;
            const int c8 = r / tpb, vox = p.bx * p.by;
            float sum[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            Ring q;
            for (int k = kbeg; k < kend; ++k, q.next(S)) {
                if (!__all_sync(0xffffffffu, mbar_wait(bar0 + 8u * q.s, q.r & 1u, kWaitLimitNs))) {
                    if (lane == 0) atomicOr(p.err, ERR_TIMEOUT);
                    ok = false;
                    break;
                }
                const uint8_t* bst = smem + (size_t)q.s * p.stage_bytes + p.a_bytes;
                for (int v = r % tpb; v < vox; v += tpb) {
                    const int y = v / p.bx, x = v % p.bx;
                    const uint4 u = *reinterpret_cast<const uint4*>(bst + (size_t)((3 * y + 1) * nb + c8) * row + 16 * x);
                    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float2 f = __bfloat1622float2(h[i]);
                        sum[2 * i] += f.x;
                        sum[2 * i + 1] += f.y;
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(bar0 + 8u * (S + q.s));
            }
            constexpr int width = tpb < 32 ? tpb : 32;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                for (int o = width / 2; o; o >>= 1) sum[i] += __shfl_xor_sync(0xffffffffu, sum[i], o);
                if (ok && lane % width == 0) atomicAdd(p.db + co0 + 8 * c8 + i, sum[i]);
            }
        }
        ok = __all_sync(0xffffffffu, ok && mbar_wait(done, 0, kWaitLimitNs));
        if (!ok) {
            if (lane == 0) atomicOr(p.err, ERR_TIMEOUT);
        } else if (kend > kbeg) {
            tc_fence_after();
            const int ci_all = 8 * (p.kc0 + p.kc1), plane0 = (src ? p.kc0 : 0) + first;
            for (int m = 0; m < NM; ++m) {
                // row group (dy, dz, plane)
                const int gr = 16 * m + (r >> 3), dy = gr / (3 * np), dz = gr / np % 3, pl = gr % np;
                const bool wrow = gr < 9 * np && pl < real;
                for (int c = 0; c < N3; c += 16) {
                    uint32_t v[16];
                    tmem_ld16(tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(m * N3 + c), v);
                    tmem_wait_ld();
                    const int dx = c / (N3 / 3), co = c % (N3 / 3);
                    if (!wrow) continue;
                    float* dst = p.dw + ((size_t)((dz * 3 + dy) * 3 + dx) * ci_all + (plane0 + pl) * 8 + (r & 7)) * p.cout +
                                 co0 + co;
                    if (p.vec) {
#pragma unroll
                        for (int e = 0; e < 16; e += 4)
                            atomicAdd(reinterpret_cast<float4*>(dst + e),
                                      make_float4(__uint_as_float(v[e]), __uint_as_float(v[e + 1]),
                                                  __uint_as_float(v[e + 2]), __uint_as_float(v[e + 3])));
                    } else {
#pragma unroll
                        for (int e = 0; e < 16; ++e) atomicAdd(dst + e, __uint_as_float(v[e]));
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, ncols);
    }
}

namespace {
template <int N3, int NM, int KPR, int RPS>
cudaError_t launch_wr(const WgradRowsParams& p, dim3 grid, size_t smem, cudaStream_t s) {
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(wgrad_rows_kernel<N3, NM, KPR, RPS>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    wgrad_rows_kernel<N3, NM, KPR, RPS><<<grid, kThreads, smem, s>>>(p);
    return cudaGetLastError();
}

// by rows per K-step: 128 voxels for nc <= 32, 64 for nc = 64 (fewer where the
// layer has fewer rows)
template <int N3, int NM>
cudaError_t launch_wr_rows(const WgradRowsParams& p, dim3 grid, size_t smem, cudaStream_t s) {
    const int rps = p.bx == 8 ? p.by / 2 : p.by;
    if (p.bx == 32) {
        if (rps == 4) return launch_wr<N3, NM, 2, 4>(p, grid, smem, s);
        if (rps == 2) return launch_wr<N3, NM, 2, 2>(p, grid, smem, s);
    } else {
        if (rps == 8) return launch_wr<N3, NM, 1, 8>(p, grid, smem, s);
        if (rps == 4) return launch_wr<N3, NM, 1, 4>(p, grid, smem, s);
    }
    return cudaErrorInvalidValue;
}
}  // namespace

cudaError_t launch_wgrad_rows(const WgradRowsParams& p, int nm, dim3 grid, size_t smem, cudaStream_t s) {
    switch (4 * p.nc / 16 + nm) {
    case 4 + 1: return launch_wr_rows<48, 1>(p, grid, smem, s);
    case 4 + 2: return launch_wr_rows<48, 2>(p, grid, smem, s);
    case 4 + 3: return launch_wr_rows<48, 3>(p, grid, smem, s);
    case 8 + 1: return launch_wr_rows<96, 1>(p, grid, smem, s);
    case 8 + 2: return launch_wr_rows<96, 2>(p, grid, smem, s);
    case 8 + 3: return launch_wr_rows<96, 3>(p, grid, smem, s);
    case 16 + 1: return launch_wr_rows<192, 1>(p, grid, smem, s);
    case 16 + 2: return launch_wr_rows<192, 2>(p, grid, smem, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace spnn
