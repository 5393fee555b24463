// Rasterisation stage (paper §3.4 with the compositing of §2.1), re-designed
// as a per-tile CUDA blend: one block per screen tile, two pixels a lane (four
// in 32-pixel tiles), front to back over the tile's depth-sorted pair list.
//
// Per pair:  a = min(0.99, sigma exp(-q/2)), q = d^T conic d, d = pixel
// centre - splat centre; a < 1/255 is skipped; C += c a T; T *= 1 - a.
//
// The splats of a tile are staged through shared memory 128 at a time: each
// thread gathers one splat record (value -> Gaussian index -> its 48-byte
// record: centre, conic, opacity, colour), converts its centre to
// tile-relative coordinates with the double-float centre (so pixel offsets
// carry no large-magnitude rounding), folds -log2(e)/2 into the conic so the
// exponent is one ex2 instruction, and computes the box of its
// opacity-aware extent (§3.4). The lanes of a 4x4 pixel sub-block (eight, or
// four in 32-pixel tiles) walk a list of the staged splats whose box reaches
// it, in step with the warp's other sub-blocks (TileGeom in ws_blend.cuh).
//
// Bound by instruction issue: 47M warp instructions on the 1080p / 1M frame.
#include "ws_blend.cuh"
#include "ws_common.cuh"
#include "ws_kernels.cuh"

namespace ws {

namespace {

constexpr int kRangeThreads = 256;

// ranges[t] = [start, end) of tile t in the sorted key list, for every tile
// (an empty tile gets start = end), in one pass over positions 0..n: at
// position i, between the tiles a of key i-1 and c of key i, tiles a+1..c
// start and tiles a..c-1 end (scan_boundaries). Keys whose tile is >= ntiles
// (none in a frame) count as past the end.
__global__ void __launch_bounds__(kRangeThreads)
k_tile_ranges(const uint64_t* __restrict__ keys, const uint32_t* __restrict__ num_keys,
              uint2* __restrict__ ranges, uint32_t ntiles) {
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const int64_t nt = (int64_t)ntiles;
    scan_boundaries<4>(
        keys, *num_keys, nt, [nt](uint64_t k) { return min((int64_t)(k >> 31), nt); },
        [&](int64_t lo, int64_t hi, uint32_t pos) {
            for (int64_t t = lo + lane; t <= hi; t += kWarp) {
                if (t >= 0 && t < hi && t < nt) ranges[t].y = pos;
                if (t > lo && t < nt) ranges[t].x = pos;
            }
        });
}

template <int TS, int PX>
__global__ void __launch_bounds__(TileGeom<TS, PX>::THREADS, fwd_min_blocks<TS>())
k_blend(const uint2* __restrict__ ranges, const uint32_t* __restrict__ order, const uint32_t* __restrict__ vals,
        const float4* __restrict__ splats, const Frame f, float* __restrict__ image, float* __restrict__ t_final, uint32_t* __restrict__ n_contrib) {
    pdl_wait();
    const FloatSplats sp{splats};
    const uint32_t t = order ? __ldg(order + blockIdx.x) : blockIdx.x;
    blend_tile<TS, PX>(f, (int)t, ranges[t], vals, sp, image, t_final, n_contrib);
}

}  // namespace

cudaError_t launch_tile_ranges(const uint64_t* keys, const uint32_t* num_keys, uint32_t* ranges, uint32_t ntiles,
                               uint32_t flags, cudaStream_t stream) {
    if (flags & WS_CFG_RANGES_GIVEN) return cudaSuccess;
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    uint2* r2w = reinterpret_cast<uint2*>(ranges);
    return launch_pdl(k_tile_ranges, dim3(sms * 8), dim3(kRangeThreads), 0, stream, keys, num_keys, r2w, ntiles);
}

cudaError_t launch_rasterize(const uint32_t* num_keys, int64_t /*key_capacity_hint*/,
                             const uint64_t* keys, const uint32_t* vals, const float* splats,
                             const Frame& f, uint32_t* ranges, const uint32_t* order, float* image, float* t_final,
                             uint32_t* n_contrib, cudaStream_t stream) {
    const int ntiles = f.TX * f.TY;
    if (ntiles == 0) return cudaSuccess;
    const cudaError_t e = launch_tile_ranges(keys, num_keys, ranges, (uint32_t)ntiles, f.flags, stream);
    if (e != cudaSuccess) return e;
    const uint2* r2 = reinterpret_cast<const uint2*>(ranges);
    const float4* s4 = reinterpret_cast<const float4*>(splats);
    auto run = [&](auto kernel, int threads) {
        return launch_pdl(kernel, dim3(ntiles), dim3(threads), 0, stream, r2, order, vals, s4, f, image, t_final,
                          n_contrib);
    };
    switch (f.TS) {
        case 8: return run(k_blend<8, tile_px<8>()>, TileGeom<8, tile_px<8>()>::THREADS);
        case 16: return run(k_blend<16, tile_px<16>()>, TileGeom<16, tile_px<16>()>::THREADS);
        case 32: return run(k_blend<32, tile_px<32>()>, TileGeom<32, tile_px<32>()>::THREADS);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace ws
