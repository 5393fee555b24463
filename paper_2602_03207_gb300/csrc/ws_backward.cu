// Deterministic backward of the render path (the paper renders only; §1
// notes the 3DGS representation is differentiable). No float atomics: every
// (tile, splat) pair owns one 9-float record of partial derivatives at its
// emission slot  offsets[g] + (ty - y0) * w + (tx - x0)  (the slot the
// compaction gave it), each record is written exactly once, and each
// Gaussian sums its contiguous records in slot order. Results are therefore
// bitwise reproducible.
//
// k_blend_bwd: one block per tile, back to front from the stored final
//   transmittance: a walk that leaves two numbers per pixel and visit, then a
//   thread per visit that sums its 16 pixels, then a thread per splat that
//   adds its visits in a fixed order (BwdPixels in ws_blend.cuh) and writes
//   the pair's record at its slot.
// k_preprocess_bwd: one thread per Gaussian: slot-ordered sum of its
//   records, then the adjoint of conic = Sigma'^{-1}, Sigma' = T Sigma T^T,
//   T = J W (J's guard-band clamp passes no gradient), the projection of
//   the centre, Sigma = M M^T with M = R(q) diag(exp(log_scale)), the
//   quaternion normalisation, sigma = sigmoid(logit) and the SH colour
//   (clamped channels pass no gradient).
#include "ws_blend.cuh"
#include "ws_common.cuh"
#include "ws_kernels.cuh"
#include "ws_project.cuh"

namespace ws {

namespace {

// Backward records of one item per block: a segment of a long list, or a tile
// in the order given (launch_tile_order); without an order the tiles
// centre-out (centre_out_tile).
template <int TS, int PX>
__global__ void __launch_bounds__(TileGeom<TS, PX>::THREADS, bwd_min_blocks<TS>())
k_blend_bwd(const uint2* __restrict__ ranges, const TileOrder order, const uint32_t* __restrict__ vals,
            const float4* __restrict__ splats, const uint2* __restrict__ rect, const uint32_t* __restrict__ offsets,
            const Frame f, const float* __restrict__ t_final, const float* __restrict__ d_image,
            const float* __restrict__ target, const PairRecords out) {
    __shared__ BwdSmem<TS, PX, bwd_batch<TS>()> sm;
    pdl_wait();
    const auto item = [&](uint32_t& t, uint32_t& first, BwdSpan& span) {
        if (order.order) return bwd_item(order, ranges, blockIdx.x, TS * TS, t, first, span);
        t = (uint32_t)centre_out_tile(f, blockIdx.x);
        const uint2 range = ranges[t];
        first = range.x;
        span = BwdSpan{0u, range.y - range.x, nullptr, 0u, 1u};
        return true;
    };
    uint32_t t, first;
    BwdSpan span;
    if (!item(t, first, span)) return;
    if (bwd_tile_body<TS, PX, true>(f, (int)t, first, span, vals, splats, rect, offsets, t_final, d_image, target, out,
                                    sm))
        return;
    // an infinite, NaN or overflowing value: the whole item again with the selecting walk
    __syncthreads();
    item(t, first, span);
    bwd_tile_body<TS, PX, false>(f, (int)t, first, span, vals, splats, rect, offsets, t_final, d_image, target, out, sm);
}

// The states of the long lists' segments, one per block (segment_state).
template <int TS, int PX>
__global__ void __launch_bounds__(TileGeom<TS, PX>::THREADS, fwd_min_blocks<TS>())
k_seg_state(const uint2* __restrict__ ranges, const TileOrder order, const uint32_t* __restrict__ vals,
            const float4* __restrict__ splats, const Frame f, const float* __restrict__ d_image,
            const float* __restrict__ target) {
    pdl_wait();
    uint32_t t, first;
    BwdSpan span;
    if (!bwd_item(order, ranges, blockIdx.x, TS * TS, t, first, span)) return;
    segment_state<TS, PX>(f, (int)t, first + span.lo, first + span.hi, vals, splats, d_image, target,
                          order.states + (size_t)blockIdx.x * (TS * TS));
}

constexpr int kPbThreads = 128;

__global__ void __launch_bounds__(kPbThreads, 8)
k_preprocess_bwd(int64_t n, const float* __restrict__ means, const float* __restrict__ log_scales,
                 const float4* __restrict__ quats, const float4* __restrict__ sh, const Frame f,
                 const float4* __restrict__ splats, const uint32_t* __restrict__ offsets, const uint32_t* __restrict__ touched,
                 uint32_t cap, const float4* __restrict__ partials, float* __restrict__ d_means,
                 float* __restrict__ d_log_scales, float4* __restrict__ d_quats,
                 float* __restrict__ d_logits, float4* __restrict__ d_sh) {
    __shared__ __align__(16) float s_sh[kPbThreads / kWarp][kWarp * kShPad];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i = (int64_t)blockIdx.x * kPbThreads + threadIdx.x;
    const bool valid = i < n;
    pdl_wait();
    const uint32_t cnt = valid ? __ldg(touched + i) : 0u;
    const bool vis = cnt > 0;

    // The SH records of this warp's visible Gaussians are copied into shared
    // memory asynchronously (16-byte copies, coalesced across the warp) while
    // the pair records are summed and the geometry adjoint runs.
    const int64_t warp_first = (int64_t)blockIdx.x * kPbThreads + warp * kWarp;
    float* stage = s_sh[warp];
    const uint32_t need = __ballot_sync(kFull, vis);
    if (need) {
        const float4* src = sh + warp_first * 12;
#pragma unroll
        for (int r = 0; r < 12; ++r) {
            const int v = lane + r * kWarp;
            const int g = v / 12, c = v - g * 12;
            if ((need >> g) & 1u) cp_async16(stage + g * kShPad + 4 * c, src + v);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }

    float gm[3] = {0.f, 0.f, 0.f}, gls[3] = {0.f, 0.f, 0.f}, gq[4] = {0.f, 0.f, 0.f, 0.f}, glogit = 0.f;
    float pr[kPart];
#pragma unroll
    for (int c = 0; c < kPart; ++c) pr[c] = 0.f;
    float X[3] = {0.f, 0.f, 0.f};
    float col[3] = {0.f, 0.f, 0.f};
    if (vis) {
        const uint32_t first = __ldg(offsets + i);
        // pairs at slots past the key capacity were dropped by the emission
        // (the frame carries WS_FLAG_CAPACITY): their records do not exist
        const uint32_t nrec = first >= cap ? 0u : min(cnt, cap - first);
        X[0] = __ldg(means + 3 * i);
        X[1] = __ldg(means + 3 * i + 1);
        X[2] = __ldg(means + 3 * i + 2);
        const float sig = __ldg(splats + kSplatVec4 * i + 1).w;
        const float4 q4 = __ldg(quats + i);
        const float ls[3] = {__ldg(log_scales + 3 * i), __ldg(log_scales + 3 * i + 1), __ldg(log_scales + 3 * i + 2)};
        const float4 cl = __ldg(splats + kSplatVec4 * i + 2);
        col[0] = cl.x;
        col[1] = cl.y;
        col[2] = cl.z;
        // slot-ordered sum of this Gaussian's pair records
        sum_pair_records(partials, reinterpret_cast<const float*>(partials + 2 * (size_t)cap), first, nrec, pr);
        glogit = pr[5] * (1.f - sig);  // pr[5] = sigma dL/dsigma
        float M[9], gM[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        gaussian_shape(q4, ls[0], ls[1], ls[2], M);
        splat_adjoint(f, X, M, pr, cl.w, gm, gM);  // cl.w: the axis basis's t
        shape_adjoint(q4, ls, gM, gls, gq);
    }

    // SH colour adjoint; gradients staged back through shared memory for
    // coalesced writes (zeros for Gaussians that are not visible).
    const int64_t avail = n - warp_first;
    const int nvec = avail <= 0 ? 0 : (int)(avail >= kWarp ? kWarp * 12 : avail * 12);
    if (need) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();
    }
    float* mine = stage + lane * kShPad;
    if (vis) {
        // the SH gradients overwrite this lane's staged coefficients in place
        // (sh_adjoint reads every coefficient before it writes a gradient)
        sh_adjoint<false>(f, X, mine, col, pr, gm, mine);
    } else if (need) {
#pragma unroll
        for (int k = 0; k < 48; ++k) mine[k] = 0.f;
    }
    if (need) {
        __syncwarp();
        float4* dst = d_sh + warp_first * 12;
#pragma unroll
        for (int r = 0; r < 12; ++r) {
            const int v = lane + r * kWarp;
            if (v < nvec) {
                const int g = v / 12, c = v - g * 12;
                dst[v] = *reinterpret_cast<const float4*>(stage + g * kShPad + 4 * c);
            }
        }
    } else {
        // no visible Gaussian in this warp: zero gradients, coalesced
        float4* dst = d_sh + warp_first * 12;
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int r = 0; r < 12; ++r) {
            const int v = lane + r * kWarp;
            if (v < nvec) dst[v] = zero;
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


// Tiles sorted by the length of their lists, longest first (64 classes, two
// per octave): a counting sort by one block, with integer atomics in shared
// memory, so that the order within a class and warp is not fixed; no result
// depends on the order that the tiles are taken in. A tile's
// time in the backward grows with its list, and a long one that starts late
// runs on alone: on the 720p / 500k step (lists up to 914, mean 138) the SMs
// were busy for 170k of the 237k cycles of the tile-centred order. The
// launch costs 4 us there and the backward call goes from 151.8 to 140.6 us.
constexpr int kOrderThreads = 1024;
constexpr int kOrderBits = 6;

__device__ __forceinline__ uint32_t length_class(uint32_t len) {
    if (len < 2u) return 63u;
    const int lz = 31 - __clz(len);
    return 63u - (uint32_t)(2 * lz + ((len >> (lz - 1)) & 1u));
}

// Lists of more than head[1] positions are cut into segments of that length
// (max_split > 0): the shortest for which max_split segments are enough, as 2
// total / max_split positions each give at most total / head[1] + (lists cut)
// of them. The total is the sum of the lengths: a caller's ranges may hold
// anything, such as (0, 0), for an empty tile.
__global__ void __launch_bounds__(kOrderThreads)
k_tile_order(const uint2* __restrict__ ranges, uint32_t ntiles, uint32_t* __restrict__ order,
             uint32_t* __restrict__ head, uint2* __restrict__ split, uint32_t max_split) {
    constexpr int W = kOrderThreads / 32, R = 1 << kOrderBits, U = 4;
    __shared__ uint32_t s_cnt[W][R];
    __shared__ uint32_t s_red[W + 1];
    __shared__ uint32_t s_split;
    __shared__ unsigned long long s_total;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < W * R; i += kOrderThreads) (&s_cnt[0][0])[i] = 0u;
    if (threadIdx.x == 0) {
        s_split = 0u;
        s_total = 0ull;
    }
    pdl_wait();
    __syncthreads();
    uint32_t seg_len = ~0u;
    unsigned long long sum = 0ull;
    const uint32_t per = (ntiles + kOrderThreads * U - 1) / (kOrderThreads * U) * (32 * U);
    const uint32_t lo = min(warp * per, ntiles), hi = min(lo + per, ntiles);
    // pass 0 counts, pass 1 places
    for (int pass = 0; pass < 2; ++pass) {
        for (uint32_t i0 = lo; i0 < hi; i0 += 32 * U) {
            uint32_t len[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t i = i0 + u * 32 + lane;
                const uint2 r = i < hi ? __ldg(ranges + i) : make_uint2(0u, 0u);
                len[u] = r.y - r.x;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t i = i0 + u * 32 + lane;
                if (i >= hi) break;
                if (!pass) sum += len[u];
                const uint32_t at = atomicAdd(&s_cnt[warp][length_class(len[u])], 1u);
                if (pass) order[at] = i;
                if (pass && len[u] > seg_len) {
                    const uint32_t nseg = (len[u] + seg_len - 1) / seg_len;
                    const uint32_t base = atomicAdd(&s_split, nseg);
                    for (uint32_t k = 0; k < nseg && base + k < max_split; ++k)
                        split[base + k] = make_uint2(i | (k << kSplitTileBits), base);
                }
            }
        }
        if (!pass && max_split) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
            if (lane == 0) atomicAdd(&s_total, sum);
        }
        __syncthreads();
        if (pass) break;
        if (max_split) {
            const unsigned long long need = (2ull * s_total + max_split - 1) / max_split;
            seg_len = max(kSplitLeast, (uint32_t)min((need + kSplitUnit - 1) / kSplitUnit * kSplitUnit, 0xffffffffull));
        }
        // counts -> first positions, by class and then warp
        static_assert(W * R == 2 * kOrderThreads, "two counters per thread");
        const int c = threadIdx.x / (W / 2), w = (threadIdx.x % (W / 2)) * 2;
        const uint32_t a = s_cnt[w][c], b = s_cnt[w + 1][c];
        uint32_t total;
        const uint32_t ex = block_exclusive_scan<kOrderThreads>(a + b, s_red, &total);
        s_cnt[w][c] = ex;
        s_cnt[w + 1][c] = ex + a;
        __syncthreads();
    }
    if (max_split && threadIdx.x == 0) {
        head[0] = s_split;
        head[1] = seg_len;
    }
}

}  // namespace

// Scratch: [pair records, 36 B per key | tile order | head | split | states],
// the last three from kSplitMinCapacity on.
size_t backward_scratch_bytes(int64_t key_capacity) {
    const int64_t cap = key_capacity > 0 ? key_capacity : 1;
    size_t bytes = (size_t)cap * kPart * sizeof(float) + 256 + kOrderMax * sizeof(uint32_t);
    if (cap >= kSplitMinCapacity) bytes += 256 + kSplitMost * sizeof(uint2) + kSplitStateBytes;
    return bytes;
}

cudaError_t launch_tile_order(const uint32_t* ranges, uint32_t ntiles, int side, int64_t key_capacity, void* scratch,
                              TileOrder* o, cudaStream_t stream) {
    *o = TileOrder{nullptr, nullptr, nullptr, nullptr, 0u};
    const int64_t cap = key_capacity > 0 ? key_capacity : 1;
    const bool cut = cap >= kSplitMinCapacity &&
                     (cap >= kSplitAnyCapacity || cap >= (int64_t)kSplitMean * (int64_t)ntiles);
    if (ntiles == 0 || ntiles > kOrderMax || (ntiles < kOrderMin && !cut)) return cudaSuccess;
    char* base = static_cast<char*>(scratch) + (((size_t)cap * kPart * sizeof(float) + 255) & ~size_t(255));
    uint32_t* order = reinterpret_cast<uint32_t*>(base);
    uint32_t* head = order + kOrderMax;
    uint2* split = reinterpret_cast<uint2*>(head + 64);
    o->order = order;
    if (cut) {
        o->head = head;
        o->split = split;
        o->states = reinterpret_cast<float2*>(split + kSplitMost);
        const size_t states = kSplitStateBytes / ((size_t)side * side * sizeof(float2));
        const uint32_t most = ntiles < kOrderMin ? kSplitMost : kSplitMost / 2;
        o->max_split = states < most ? (uint32_t)states : most;
    }
    return launch_pdl(k_tile_order, dim3(1), dim3(kOrderThreads), 0, stream, reinterpret_cast<const uint2*>(ranges),
                      ntiles, order, head, split, o->max_split);
}

cudaError_t launch_backward(int64_t n, const float* means, const float* log_scales, const float* quats,
                            const float* sh, const Frame& f, const float* splats, const uint16_t* rect,
                            const uint32_t* offsets, const uint32_t* tiles_touched,
                            const uint32_t* vals, const uint32_t* ranges, const TileOrder& order, const float* t_final,
                            const float* d_image, const float* target, float* d_means,
                            float* d_log_scales, float* d_quats, float* d_logits, float* d_sh,
                            int64_t key_capacity, void* scratch, cudaStream_t stream) {
    const PairRecords partials = pair_records(scratch, key_capacity);
    const int ntiles = f.TX * f.TY;
    const uint2* r2 = reinterpret_cast<const uint2*>(ranges);
    const float4* s4 = reinterpret_cast<const float4*>(splats);
    const uint2* rc = reinterpret_cast<const uint2*>(rect);
    cudaError_t e = cudaSuccess;
    if (ntiles > 0) {
        auto run = [&](auto states, auto kernel, int threads) {
            if (order.max_split) {
                const cudaError_t se = launch_pdl(states, dim3(order.max_split), dim3(threads), 0, stream, r2, order,
                                                  vals, s4, f, d_image, target);
                if (se != cudaSuccess) return se;
            }
            return launch_pdl(kernel, dim3(ntiles + order.max_split), dim3(threads), 0, stream, r2, order, vals, s4,
                              rc, offsets, f, t_final, d_image, target, partials);
        };
        constexpr int P8 = tile_px<8>(), P16 = tile_px<16>(), P32 = tile_px<32>();
        switch (f.TS) {
            case 8: e = run(k_seg_state<8, P8>, k_blend_bwd<8, P8>, TileGeom<8, P8>::THREADS); break;
            case 16: e = run(k_seg_state<16, P16>, k_blend_bwd<16, P16>, TileGeom<16, P16>::THREADS); break;
            case 32: e = run(k_seg_state<32, P32>, k_blend_bwd<32, P32>, TileGeom<32, P32>::THREADS); break;
            default: return cudaErrorInvalidValue;
        }
        if (e != cudaSuccess) return e;
    }
    if (n > 0) {
        const int64_t blocks = (n + kPbThreads - 1) / kPbThreads;
        e = launch_pdl(k_preprocess_bwd, dim3((unsigned)blocks), dim3(kPbThreads), 0, stream, n, means, log_scales,
                       reinterpret_cast<const float4*>(quats), reinterpret_cast<const float4*>(sh), f, s4,
                       offsets, tiles_touched, (uint32_t)key_capacity, (const float4*)partials.p8, d_means, d_log_scales,
                       reinterpret_cast<float4*>(d_quats), d_logits, reinterpret_cast<float4*>(d_sh));
    }
    return e;
}

}  // namespace ws
