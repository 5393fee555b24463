// Many views of one scene as one batch: the same per-Gaussian projection,
// per-tile blend and adjoint as the single-view path (shared device code, so
// every view's image is bit-identical to rendering it alone), organised so
// the scene is read once for all views.
//
//   k_preprocess_batch   one thread per Gaussian; its inputs (236 B, SH
//                        staged in shared memory) are read once and every
//                        view is projected from registers; outputs are
//                        view-major and written coalesced per view.
//   compaction / sort    the single-view kernels over V*n items, with tile
//                        ids offset into one global tile grid, so one sort
//                        orders every view's (tile, depth) keys.
//   k_blend_batch        one launch over every (view, tile) work item.
//   k_blend_bwd_batch    likewise, longest lists first, records at each pair's
//                        emission slot.
//   k_preprocess_bwd_batch  one thread per Gaussian: for each view in order,
//                        the slot-ordered sum of its records and that view's
//                        adjoint, accumulated in view order (deterministic).
#include "ws_blend.cuh"
#include "ws_common.cuh"
#include "ws_kernels.cuh"
#include "ws_project.cuh"

namespace ws {

namespace {

constexpr int kBatchThreads = 128;

__global__ void __launch_bounds__(kBatchThreads)
k_preprocess_batch(int64_t n, const float* __restrict__ means, const float* __restrict__ log_scales,
                   const float4* __restrict__ quats, const float* __restrict__ logits,
                   const float4* __restrict__ sh, const FrameTable ft, float4* __restrict__ splats,
                   float* __restrict__ depth, uint2* __restrict__ rect, uint32_t* __restrict__ tiles_touched) {
    __shared__ __align__(16) float s_sh[kBatchThreads / kWarp][kWarp * kShPad];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i = (int64_t)blockIdx.x * kBatchThreads + threadIdx.x;
    const bool valid = i < n;
    const int64_t warp_first = (int64_t)blockIdx.x * kBatchThreads + warp * kWarp;
    pdl_wait();

    float logit = 0.f, x = 0.f, y = 0.f, z = 0.f, l0 = 0.f, l1 = 0.f, l2 = 0.f;
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
    if (valid) {
        logit = __ldg(logits + i);
        x = __ldg(means + 3 * i);
        y = __ldg(means + 3 * i + 1);
        z = __ldg(means + 3 * i + 2);
        q = __ldg(quats + i);
        l0 = __ldg(log_scales + 3 * i);
        l1 = __ldg(log_scales + 3 * i + 1);
        l2 = __ldg(log_scales + 3 * i + 2);
    }
    const bool opaque_enough = valid && passes_opacity(ft.f[0], logit);
    const uint32_t need = __ballot_sync(kFull, opaque_enough);
    float* stage = s_sh[warp];
    if (need) {
        const float4* src = sh + warp_first * 12;
#pragma unroll
        for (int r = 0; r < 12; ++r) {
            const int v = lane + r * kWarp;
            const int g = v / 12, c = v - g * 12;
            if ((need >> g) & 1u) cp_async16(stage + g * kShPad + 4 * c, src + v);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();
    }
    // what the views share (the configuration's flags are every view's)
    float M[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, sigma = 0.f, qc = 0.f;
    const bool drawable = opaque_enough && gaussian_shape(q, l0, l1, l2, M);
    if (drawable) qc = opacity_extent(ft.f[0], logit, sigma);
    for (int v = 0; v < ft.views; ++v) {
        const Frame& f = ft.f[v];
        const int64_t o = (int64_t)v * n + i;
        bool vis = false;
        Projection P;
        if (valid) {
            const float d = view_depth(f, x, y, z);
            depth[o] = d;
            vis = drawable && d > f.znear && project_splat(f, x, y, z, M, sigma, qc, P);
        }
        float3 c3 = make_float3(0.f, 0.f, 0.f);
        if (vis) {
            const float dx = x - f.campos[0], dy = y - f.campos[1], dz = z - f.campos[2];
            const float inv = rsqrtf(dx * dx + dy * dy + dz * dz);
            sh_eval(dx * inv, dy * inv, dz * inv, stage + lane * kShPad, c3);
        }
        // every lane stores its entries (zeros where culled): whole sectors
        if (valid) {
            store_splat(splats + kSplatVec4 * o, vis, P, c3);
            rect[o] = vis ? make_uint2(P.x0 | (P.y0 << 16), P.x1 | (P.y1 << 16)) : make_uint2(0u, 0u);
            tiles_touched[o] = vis ? (P.x1 - P.x0 + 1) * (P.y1 - P.y0 + 1) : 0u;
        }
    }
}

template <int TS, int PX>
__global__ void __launch_bounds__(TileGeom<TS, PX>::THREADS, fwd_min_blocks<TS>())
k_blend_batch(const uint2* __restrict__ ranges, const uint32_t* __restrict__ order,
              const uint32_t* __restrict__ vals, int64_t n, const float4* __restrict__ splats, const FrameTable ft,
              float* __restrict__ image, float* __restrict__ t_final, uint32_t* __restrict__ n_contrib) {
    pdl_wait();
    const uint32_t t = order ? __ldg(order + blockIdx.x) : blockIdx.x;
    const int v = view_of_tile(ft.tile_off, ft.views, t);
    const uint64_t vo = (uint64_t)v * (uint64_t)n, po = ft.pix_off[v];
    const FloatSplats sp{splats + kSplatVec4 * vo};
    blend_tile<TS, PX>(ft.f[v], (int)(t - ft.tile_off[v]), ranges[t], vals, sp, image + 3 * po, t_final + po,
                   n_contrib + po);
}

// Backward records of every item (a segment of a long list, or a tile of a
// view: bwd_item). PERSISTENT = false: one block per item. PERSISTENT = true: a
// grid of as many blocks as fit on the GPU at once, block b taking items b, b +
// G, b + 2G, ... (G = the grid size), so the assignment is static; no block
// waits on another.
template <int TS, int PX, bool PERSISTENT>
__global__ void __launch_bounds__(TileGeom<TS, PX>::THREADS, bwd_min_blocks<TS>())
k_blend_bwd_batch(const uint2* __restrict__ ranges, const TileOrder order, const uint32_t* __restrict__ vals,
                  int64_t n, const float4* __restrict__ splats, const uint2* __restrict__ rect,
                  const uint32_t* __restrict__ offsets, const FrameTable ft, const float* __restrict__ t_final,
                  const float* __restrict__ d_image, const float* __restrict__ target, const PairRecords out) {
    __shared__ BwdSmem<TS, PX, bwd_batch<TS>()> sm;
    pdl_wait();
    const uint32_t items = ft.tile_off[ft.views] + order.max_split;
    const uint32_t stride = PERSISTENT ? gridDim.x : items;
    for (uint32_t i = blockIdx.x; i < items; i += stride) {
        const auto walk = [&](auto finite) {
            uint32_t t, first;
            BwdSpan span;
            if (!bwd_item(order, ranges, i, TS * TS, t, first, span)) return true;
            const int v = view_of_tile(ft.tile_off, ft.views, t);
            const uint64_t vo = (uint64_t)v * (uint64_t)n, po = ft.pix_off[v];
            return bwd_tile_body<TS, PX, decltype(finite)::value>(
                ft.f[v], (int)(t - ft.tile_off[v]), first, span, vals, splats + kSplatVec4 * vo, rect + vo,
                offsets + vo, t_final + po, d_image + 3 * po, target ? target + 3 * po : nullptr, out, sm);
        };
        if (!walk(std::true_type{})) {  // an infinite, NaN or overflowing value: the item again, selecting
            __syncthreads();
            walk(std::false_type{});
        }
        if (PERSISTENT) __syncthreads();  // the last reads of sm before the next item's writes
    }
}

// The states of the long lists' segments, one per block (segment_state).
template <int TS, int PX>
__global__ void __launch_bounds__(TileGeom<TS, PX>::THREADS, fwd_min_blocks<TS>())
k_seg_state_batch(const uint2* __restrict__ ranges, const TileOrder order, const uint32_t* __restrict__ vals,
                  int64_t n, const float4* __restrict__ splats, const FrameTable ft,
                  const float* __restrict__ d_image, const float* __restrict__ target) {
    pdl_wait();
    uint32_t t, first;
    BwdSpan span;
    if (!bwd_item(order, ranges, blockIdx.x, TS * TS, t, first, span)) return;
    const int v = view_of_tile(ft.tile_off, ft.views, t);
    const uint64_t vo = (uint64_t)v * (uint64_t)n, po = ft.pix_off[v];
    segment_state<TS, PX>(ft.f[v], (int)(t - ft.tile_off[v]), first + span.lo, first + span.hi, vals,
                          splats + kSplatVec4 * vo, d_image + 3 * po, target ? target + 3 * po : nullptr,
                          order.states + (size_t)blockIdx.x * (TS * TS));
}

__global__ void __launch_bounds__(kBatchThreads)
k_preprocess_bwd_batch(int64_t n, const float* __restrict__ means, const float* __restrict__ log_scales,
                       const float4* __restrict__ quats, const float4* __restrict__ sh, const FrameTable ft,
                       const float4* __restrict__ splats, const uint32_t* __restrict__ offsets,
                       const uint32_t* __restrict__ touched,
                       uint32_t cap, const float4* __restrict__ partials, float* __restrict__ d_means,
                       float* __restrict__ d_log_scales, float4* __restrict__ d_quats,
                       float* __restrict__ d_logits, float4* __restrict__ d_sh) {
    __shared__ __align__(16) float s_sh[kBatchThreads / kWarp][kWarp * kShPad];
    __shared__ __align__(16) float s_gsh[kBatchThreads / kWarp][kWarp * kShPad];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i = (int64_t)blockIdx.x * kBatchThreads + threadIdx.x;
    const bool valid = i < n;
    const int64_t warp_first = (int64_t)blockIdx.x * kBatchThreads + warp * kWarp;
    const int64_t avail = n - warp_first;
    const int nvec = avail <= 0 ? 0 : (int)(avail >= kWarp ? kWarp * 12 : avail * 12);
    pdl_wait();

    float X[3] = {0.f, 0.f, 0.f}, ls[3] = {0.f, 0.f, 0.f};
    float4 q4 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (valid) {
        X[0] = __ldg(means + 3 * i);
        X[1] = __ldg(means + 3 * i + 1);
        X[2] = __ldg(means + 3 * i + 2);
        ls[0] = __ldg(log_scales + 3 * i);
        ls[1] = __ldg(log_scales + 3 * i + 1);
        ls[2] = __ldg(log_scales + 3 * i + 2);
        q4 = __ldg(quats + i);
    }
    // stage this warp's SH coefficients; zero the SH gradient accumulators
    float* stage = s_sh[warp];
    float* gsh = s_gsh[warp] + lane * kShPad;
    {
        const float4* src = sh + warp_first * 12;
#pragma unroll
        for (int r = 0; r < 12; ++r) {
            const int v = lane + r * kWarp;
            if (v < nvec) {
                const int g = v / 12, c = v - g * 12;
                *reinterpret_cast<float4*>(stage + g * kShPad + 4 * c) = __ldg(src + v);
            }
        }
#pragma unroll
        for (int k = 0; k < 48; ++k) gsh[k] = 0.f;
        __syncwarp();
    }
    float gm[3] = {0.f, 0.f, 0.f}, gsig = 0.f;
    float M[9], gM[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (valid) gaussian_shape(q4, ls[0], ls[1], ls[2], M);
    int64_t last_seen = -1;  // this Gaussian in the last view that sees it
    // A view's pair count and first slot are loaded two views ahead and its
    // colour before its records, so that their latencies overlap the adjoints
    // (15 warps an SM, the SH accumulators allow no more): 64 views of 2M 3.96 ->
    // 3.61 ms against one view ahead and the colour after the records; prefetches
    // of the next view's records gave 1 % more and are left out.
    const float* p9 = reinterpret_cast<const float*>(partials + 2 * (size_t)cap);
    uint32_t cnt_next = valid ? __ldg(touched + i) : 0u;
    uint32_t off_next = valid ? __ldg(offsets + i) : 0u;
    uint32_t cnt_then = valid && ft.views > 1 ? __ldg(touched + n + i) : 0u;
    uint32_t off_then = valid && ft.views > 1 ? __ldg(offsets + n + i) : 0u;
    for (int v = 0; v < ft.views; ++v) {
        const int64_t o = (int64_t)v * n + i;
        const uint32_t cnt = cnt_next, first = off_next;
        cnt_next = cnt_then;
        off_next = off_then;
        if (valid && v + 2 < ft.views) {
            cnt_then = __ldg(touched + o + 2 * n);
            off_then = __ldg(offsets + o + 2 * n);
        }
        if (cnt == 0) continue;
        const float4 cl = __ldg(splats + kSplatVec4 * o + 2);  // colour and the axis basis's t
        last_seen = o;
        float pr[kPart];
#pragma unroll
        for (int c = 0; c < kPart; ++c) pr[c] = 0.f;
        // records past the key capacity were never written (the emission
        // dropped those pairs and raised WS_FLAG_CAPACITY)
        const uint32_t nrec = first >= cap ? 0u : min(cnt, cap - first);
        sum_pair_records(partials, p9, first, nrec, pr);
        gsig += pr[5];  // sigma dL/dsigma
        const Frame& f = ft.f[v];
        splat_adjoint(f, X, M, pr, cl.w, gm, gM);
        const float col[3] = {cl.x, cl.y, cl.z};
        sh_adjoint<true>(f, X, stage + lane * kShPad, col, pr, gm, gsh);
    }
    float gls[3] = {0.f, 0.f, 0.f}, gq[4] = {0.f, 0.f, 0.f, 0.f};
    float glogit = 0.f;
    if (last_seen >= 0) {
        shape_adjoint(q4, ls, gM, gls, gq);
        glogit = gsig * (1.f - __ldg(splats + kSplatVec4 * last_seen + 1).w);  // sigma: the same in every view
    }
    __syncwarp();
    float4* dst = d_sh + warp_first * 12;
    const float* gstage = s_gsh[warp];
#pragma unroll
    for (int r = 0; r < 12; ++r) {
        const int v = lane + r * kWarp;
        if (v < nvec) {
            const int g = v / 12, c = v - g * 12;
            dst[v] = *reinterpret_cast<const float4*>(gstage + g * kShPad + 4 * c);
        }
    }
    if (valid) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            d_means[3 * i + a] = gm[a];
            d_log_scales[3 * i + a] = gls[a];
        }
        d_quats[i] = make_float4(gq[0], gq[1], gq[2], gq[3]);
        d_logits[i] = glogit;
    }
}

__global__ void k_residual(int64_t count, const float4* __restrict__ image, const float4* __restrict__ target,
                           float4* __restrict__ d_image, int64_t count4) {
    pdl_wait();
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < count4; j += (int64_t)gridDim.x * blockDim.x) {
        const float4 a = __ldg(image + j), b = __ldg(target + j);
        d_image[j] = make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
    }
    // tail (count not a multiple of 4)
    if (blockIdx.x == 0 && threadIdx.x < (count & 3)) {
        const int64_t k = count4 * 4 + threadIdx.x;
        reinterpret_cast<float*>(d_image)[k] =
            reinterpret_cast<const float*>(image)[k] - reinterpret_cast<const float*>(target)[k];
    }
}

}  // namespace

cudaError_t launch_preprocess_batch(int64_t n, const float* means, const float* log_scales, const float* quats,
                                    const float* logits, const float* sh, const FrameTable& ft, float* splats,
                                    float* depth, uint16_t* rect, uint32_t* tiles_touched, cudaStream_t stream) {
    if (n == 0) return cudaSuccess;
    const int64_t blocks = (n + kBatchThreads - 1) / kBatchThreads;
    return launch_pdl(k_preprocess_batch, dim3((unsigned)blocks), dim3(kBatchThreads), 0, stream, n, means,
                      log_scales, reinterpret_cast<const float4*>(quats), logits, reinterpret_cast<const float4*>(sh),
                      ft, reinterpret_cast<float4*>(splats), depth, reinterpret_cast<uint2*>(rect), tiles_touched);
}

cudaError_t launch_rasterize_batch(const uint32_t* num_keys, const uint64_t* keys, const uint32_t* vals, int64_t n,
                                   const float* splats, const FrameTable& ft, uint32_t* ranges, const uint32_t* order,
                                   float* image, float* t_final, uint32_t* n_contrib, cudaStream_t stream) {
    const uint32_t ntiles = ft.tile_off[ft.views];
    if (ntiles == 0) return cudaSuccess;
    const cudaError_t e = launch_tile_ranges(keys, num_keys, ranges, ntiles, ft.f[0].flags, stream);
    if (e != cudaSuccess) return e;
    const uint2* r2 = reinterpret_cast<const uint2*>(ranges);
    const float4* s4 = reinterpret_cast<const float4*>(splats);
    auto run = [&](auto kernel, int threads) {
        return launch_pdl(kernel, dim3(ntiles), dim3(threads), 0, stream, r2, order, vals, n, s4, ft, image,
                          t_final, n_contrib);
    };
    switch (ft.f[0].TS) {
        case 8: return run(k_blend_batch<8, tile_px<8>()>, TileGeom<8, tile_px<8>()>::THREADS);
        case 16: return run(k_blend_batch<16, tile_px<16>()>, TileGeom<16, tile_px<16>()>::THREADS);
        case 32: return run(k_blend_batch<32, tile_px<32>()>, TileGeom<32, tile_px<32>()>::THREADS);
        default: return cudaErrorInvalidValue;
    }
}

template <int TS>
cudaError_t launch_bwd_items(const uint2* r2, const TileOrder& order, const uint32_t* vals, int64_t n, const float4* s4,
                             const uint2* rc, const uint32_t* offsets, const FrameTable& ft, const float* t_final,
                             const float* d_image, const float* target, const PairRecords& out, bool persistent, cudaStream_t stream) {
    const uint32_t items = ft.tile_off[ft.views] + order.max_split;
    constexpr int PX = tile_px<TS>();
    constexpr int kThreads = TileGeom<TS, PX>::THREADS;
    cudaError_t e = cudaSuccess;
    if (order.max_split) {
        e = launch_pdl(k_seg_state_batch<TS, PX>, dim3(order.max_split), dim3(kThreads), 0, stream, r2, order, vals, n,
                       s4, ft, d_image, target);
        if (e != cudaSuccess) return e;
    }
    if (!persistent)
        return launch_pdl(k_blend_bwd_batch<TS, PX, false>, dim3(items), dim3(kThreads), 0, stream, r2, order, vals, n,
                          s4, rc, offsets, ft, t_final, d_image, target, out);
    int dev = 0, sms = 148, occ = 1;
    e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_blend_bwd_batch<TS, PX, true>, kThreads, 0);
    if (e != cudaSuccess) return e;
    const uint32_t grid = min(items, (uint32_t)(sms * (occ > 0 ? occ : 1)));
    return launch_pdl(k_blend_bwd_batch<TS, PX, true>, dim3(grid), dim3(kThreads), 0, stream, r2, order, vals, n, s4,
                      rc, offsets, ft, t_final, d_image, target, out);
}

cudaError_t launch_backward_batch(int64_t n, const float* means, const float* log_scales, const float* quats,
                                  const float* sh, const FrameTable& ft, const float* splats, const uint16_t* rect,
                                  const uint32_t* offsets, const uint32_t* tiles_touched, const uint32_t* vals,
                                  const uint32_t* ranges, const TileOrder& order, const float* t_final,
                                  const float* d_image, const float* target, float* d_means,
                                  float* d_log_scales, float* d_quats, float* d_logits, float* d_sh,
                                  int64_t key_capacity, bool persistent, void* scratch, cudaStream_t stream) {
    const PairRecords partials = pair_records(scratch, key_capacity);
    const uint32_t ntiles = ft.tile_off[ft.views];
    const uint2* r2 = reinterpret_cast<const uint2*>(ranges);
    const float4* s4 = reinterpret_cast<const float4*>(splats);
    const uint2* rc = reinterpret_cast<const uint2*>(rect);
    cudaError_t e = cudaSuccess;
    if (ntiles > 0) {
        auto run = [&](auto items) {
            return items(r2, order, vals, n, s4, rc, offsets, ft, t_final, d_image, target, partials,
                         persistent, stream);
        };
        switch (ft.f[0].TS) {
            case 8: e = run(launch_bwd_items<8>); break;
            case 16: e = run(launch_bwd_items<16>); break;
            case 32: e = run(launch_bwd_items<32>); break;
            default: return cudaErrorInvalidValue;
        }
        if (e != cudaSuccess) return e;
    }
    if (n > 0) {
        const int64_t blocks = (n + kBatchThreads - 1) / kBatchThreads;
        e = launch_pdl(k_preprocess_bwd_batch, dim3((unsigned)blocks), dim3(kBatchThreads), 0, stream, n, means,
                       log_scales, reinterpret_cast<const float4*>(quats), reinterpret_cast<const float4*>(sh), ft, s4,
                       offsets, tiles_touched, (uint32_t)key_capacity, (const float4*)partials.p8, d_means,
                       d_log_scales,
                       reinterpret_cast<float4*>(d_quats), d_logits, reinterpret_cast<float4*>(d_sh));
    }
    return e;
}

cudaError_t launch_residual(int64_t count, const float* image, const float* target, float* d_image,
                            cudaStream_t stream) {
    if (count == 0) return cudaSuccess;
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return launch_pdl(k_residual, dim3(sms * 4), dim3(256), 0, stream, count,
                      reinterpret_cast<const float4*>(image), reinterpret_cast<const float4*>(target),
                      reinterpret_cast<float4*>(d_image), count / 4);
}

}  // namespace ws
