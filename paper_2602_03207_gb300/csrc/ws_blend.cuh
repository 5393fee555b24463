// Per-tile blend bodies (paper §3.4 with §2.1's compositing) shared by the
// single-view and batched kernels: the forward composite and its
// deterministic adjoint.
//
// Both are bound by instruction issue and by the latency of a step's chain
// (list entry, record, log-alpha, exponential), not by memory: on the 1080p
// / 1M frame the forward moves 63 MB in 65 us. Measured against the walk that
// they replace (two streams of 16 lanes, one pixel per lane, a bit set per
// 32 splats; the backward's partials summed by 12 shuffles a visit and 16
// selects a splat), warm, at 16-pixel tiles:
//   forward, 1080p / 1M                 80.4 -> 62.4 us (72.0M -> 47M warp instructions)
//   forward, 2160p / 6M                617.6 -> 448 us
//   backward call, 720p / 500k         220.4 -> 133 us (102.6M -> 48.7M)
//   backward call, 64 views of 2M       33.2 -> 20.1 ms
#pragma once

#include <type_traits>

#include "ws_common.cuh"

namespace ws {

constexpr int kPart = 9;  // partials of a pair: dmean x, y; dconic a, b, c; sigma dsigma; drgb r, g, b

// Whether a value may enter the backward's multiplying walk (BwdPixels), where
// a pixel that does not composite a splat adds 0 times what lies there: not
// NaN, not infinite, and small enough that no product on the way overflows:
// colour . dL/dC < 3 2^120, its distance from a b below 2^122 < 2^123.
constexpr float kWalkMost = 0x1p60f, kBehindMost = 0x1p122f;
__device__ __forceinline__ bool walkable(float x) { return fabsf(x) < kWalkMost; }

// Shared-memory record of one staged splat (48 bytes):
//   geo  = minus the tile-relative centre (-x, -y); conic premultiplied
//          A = -log2(e) a / 2, B = -log2(e) b
//   geo2 = C = -log2(e) c / 2, L = log2(sigma); the splat's axis basis
//          e1 = (ct, st) (axis_basis; staged for the backward only)
//   col  = r, g, b; 0
// The forward reads geo, geo2.xy and col.xyz; the backward everything.
struct SplatRec {
    float4 geo;
    float4 geo2;
    float4 col;
};

// Writes the null splat at index `batch` of a staging area: zero conic,
// L = -inf, so its log-alpha is -inf and it is never composited. The visit
// lists of a warp's streams are padded with it.
__device__ __forceinline__ void init_null_splat(SplatRec* s_rec, int batch) {
    if (threadIdx.x == 0) {
        s_rec[batch].geo = make_float4(0.f, 0.f, 0.f, 0.f);
        s_rec[batch].geo2 = make_float4(0.f, -INFINITY, 0.f, 0.f);
        s_rec[batch].col = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// Two floats in one 64-bit register pair, for the two-wide FP32
// instructions (each half rounds as the scalar instruction does).
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 pack2(float lo, float hi) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ F2 dup2(float x) { return pack2(x, x); }
__device__ __forceinline__ void unpack2(F2 a, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v));
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ float sum2(F2 a) {
    float lo, hi;
    unpack2(a, lo, hi);
    return __fadd_rn(lo, hi);
}

// Per-splat inputs of the blend, read from the splat records of
// ws_preprocess (three 16-byte loads of one 48-byte record): the double-float
// centre (made tile-relative without large-magnitude rounding), the conic
// (a, b, c), sigma and the colour.
struct FloatSplats {
    const float4* __restrict__ rec;
    __device__ __forceinline__ void load(uint32_t g, float ox, float oy, float& x, float& y, float& a, float& b,
                                         float& c, float& op, float4& col) const {
        const float4 m = __ldg(rec + kSplatVec4 * g);
        const float4 k = __ldg(rec + kSplatVec4 * g + 1);
        col = __ldg(rec + kSplatVec4 * g + 2);
        x = __fadd_rn(__fsub_rn(m.x, ox), m.z);
        y = __fadd_rn(__fsub_rn(m.y, oy), m.w);
        a = k.x;
        b = k.y;
        c = k.z;
        op = k.w;
    }
};

// Geometry of a TS x TS tile: its 4x4 pixel sub-blocks (numbered row-major,
// SPR per row) are the unit of culling, and a stream of 16 / PX lanes walks
// the splats that reach one sub-block, PX pixels of a column per lane. A
// warp runs SPW streams in lockstep, each on its own visit list.
//
// Why streams of few lanes: the steps a warp takes are the longest of its
// streams' lists, and the work around a pixel evaluation (the list entry,
// the three record loads, the loop, and in the backward the sum over the
// sub-block) is paid per step, so PX pixels per lane pay it once for PX
// evaluations, two of which share each FP32 instruction. On the 1080p / 1M
// frame (counted on the host): 1.68M steps with two streams of 16 lanes
// kept in step every 32 splats, 0.45M with eight streams of four lanes over a
// whole staged batch, with 7 % more (idle included) evaluations.
template <int TS, int PX>
struct TileGeom {
    static constexpr int SPR = TS / 4;
    static constexpr int NSB = SPR * SPR;
    static constexpr int LPS = 16 / PX;
    static constexpr int SPW = 32 / LPS;
    static constexpr int WARPS = NSB / SPW;
    static constexpr int THREADS = 32 * WARPS;
    static_assert(NSB % SPW == 0 && PX % 2 == 0, "whole warps of streams, pairs of pixels");
    using Mask = typename std::conditional<(NSB > 32), unsigned long long, uint32_t>::type;
    // this lane's sub-block and its pixels (tile-relative centres): column
    // px, rows py0 .. py0 + PX - 1
    __device__ static __forceinline__ int sub_block(int warp, int lane) { return warp * SPW + lane / LPS; }
    __device__ static __forceinline__ void pixel(int warp, int lane, int& ix, int& iy0) {
        const int sb = sub_block(warp, lane), q = lane % LPS;
        ix = (sb % SPR) * 4 + (q & 3);
        iy0 = (sb / SPR) * 4 + (q >> 2) * PX;
    }
};

// Pixels per lane: two (four streams a warp, four warps for a 16-pixel
// tile). Four (eight streams, two warps) execute 20 % fewer instructions but
// leave a tile of many splats to two warps: 78 against 65 us on the 1080p /
// 1M frame, whose longest list has 1,300 splats, 457 against 448 us at 2160p
// / 6M. A 32-pixel tile has enough sub-blocks for eight warps of four.
template <int TS>
__host__ __device__ constexpr int tile_px() { return TS == 32 ? 4 : 2; }

// Splats the forward stages in shared memory at a time. The visit lists hold
// 8-bit indices, the null splat's (the batch size) among them. 192 instead of
// 128: 66.3 against 64.9 us at 1080p / 1M (fewer blocks fit an SM).
template <int TS>
__host__ __device__ constexpr int fwd_batch() { return 128; }

// Blocks per SM that the blends are compiled for (their register budget). At
// 16-pixel tiles nine for the forward (56 registers: 64.9 us at 1080p / 1M
// against 65.5 with ten, 67.5 with 80 registers and 77 with 40) and six for
// the backward (80 registers: 133 us on the 720p call against 142 with the
// compiler's own choice of 72, and 140 with 127).
template <int TS>
__host__ __device__ constexpr int fwd_min_blocks() { return TS == 8 ? 16 : (TS == 16 ? 9 : 4); }
template <int TS>
__host__ __device__ constexpr int bwd_min_blocks() { return TS == 8 ? 12 : (TS == 16 ? 6 : 2); }

// One row of visit indices per stream: the batch and a padded end.
template <int BATCH>
__host__ __device__ constexpr int list_row() { return BATCH + 16; }

// Builds the visit lists of this warp's streams over the staged splats
// [lo, hi): for each stream the indices whose mask has its sub-block, in
// list order (REV: back to front), padded with the null splat. Returns the
// longest list's length. A list of the whole span rather than one bit set
// per 32 splats: the streams then wait for each other only at its end.
template <typename G, int BATCH, bool REV>
__device__ __forceinline__ int build_lists(const typename G::Mask* s_mask, int lo, int hi, uint8_t* rows, int warp,
                                           int lane) {
    constexpr int ROW = list_row<BATCH>();
    static_assert(BATCH < 256 && ROW % 16 == 0, "8-bit indices, 16-byte rows");
    constexpr uint32_t kNull4 = 0x01010101u * (uint32_t)BATCH;
    const int q = lane % G::LPS;
    uint4* mine = reinterpret_cast<uint4*>(rows + (lane / G::LPS) * ROW);
    for (int v = q; v <= (hi - lo) >> 4; v += G::LPS) mine[v] = make_uint4(kNull4, kNull4, kNull4, kNull4);
    __syncwarp();
    const uint32_t lt = lanemask_lt();
    const int sb0 = warp * G::SPW;
    int c[G::SPW];
#pragma unroll
    for (int t = 0; t < G::SPW; ++t) c[t] = 0;
    for (int k = 0; k < hi - lo; k += 32) {
        const bool in = k + lane < hi - lo;
        const int j = REV ? hi - 1 - k - lane : lo + k + lane;
        const uint32_t m = in ? (uint32_t)(s_mask[j] >> sb0) : 0u;
#pragma unroll
        for (int t = 0; t < G::SPW; ++t) {
            const bool bit = (m >> t) & 1u;
            const uint32_t bal = __ballot_sync(kFull, bit);
            if (bit) rows[t * ROW + c[t] + __popc(bal & lt)] = (uint8_t)j;
            c[t] += __popc(bal);
        }
    }
    __syncwarp();
    int steps = 0;
#pragma unroll
    for (int t = 0; t < G::SPW; ++t) steps = max(steps, c[t]);
    return steps;
}

// Bitmask of a tile's 4x4 sub-blocks whose pixel centres meet the box
// [xl, xh] x [yl, yh] (tile-relative): one compare pair per sub-block column
// and per sub-block row.
template <int SPR, typename MaskT>
__device__ __forceinline__ MaskT box_subblock_mask(float xl, float xh, float yl, float yh) {
    MaskT cols = 0;
#pragma unroll
    for (int c = 0; c < SPR; ++c)
        cols |= (xl <= (float)(c * 4) + 3.5f && xh >= (float)(c * 4) + 0.5f) ? (MaskT(1) << c) : MaskT(0);
    MaskT mask = 0;
#pragma unroll
    for (int r = 0; r < SPR; ++r)
        mask |= (yl <= (float)(r * 4) + 3.5f && yh >= (float)(r * 4) + 0.5f) ? (cols << (r * SPR)) : MaskT(0);
    return mask;
}

// Sub-blocks of columns [c_lo, c_hi] (clamped into [0, SPR)) as SPR bits:
// c_lo = ceil((xl - 3.5) / 4), c_hi = floor((xh - 0.5) / 4), the columns
// whose pixel centres 4c + 0.5 .. 4c + 3.5 meet [xl, xh].
template <int SPR>
__device__ __forceinline__ uint32_t span_bits(float xl, float xh) {
    const int lo = (int)ceilf(fmaxf((xl - 3.5f) * 0.25f, 0.f));
    const int hi = (int)floorf(fminf((xh - 0.5f) * 0.25f, (float)(SPR - 1)));
    return lo <= hi ? (2u << hi) - (1u << lo) : 0u;
}

// Bitmask of a tile's 4x4 sub-blocks that the ellipse q(dx, dy) =
// a dx^2 + 2 b dx dy + c dy^2 <= qm around the tile-relative centre (gx, gy)
// meets, one row of sub-blocks (a band of 4 pixel rows) at a time. Within
// the band the ellipse's dy runs over [u0, u1] (the band cut to the
// ellipse's half-height ey) and at height dy its x range is
// gx + (-b dy -/+ s(dy)) / a with s(dy) = sqrt(a qm - det dy^2); the left end
// is convex in dy and smallest at dy = b sqrt(qm / (det c)), the right end
// concave and largest at the opposite dy, so the band's x range is those two
// ends with dy clamped into [u0, u1]. The part of the ellipse in the band is
// convex, so it meets a sub-block of the band exactly when its x range meets
// the sub-block's columns.
template <int SPR, typename MaskT>
__device__ __forceinline__ MaskT ellipse_subblock_mask(float gx, float gy, float a, float b, float c, float qm,
                                                       float rdet, float ey, float xmargin) {
    const int r_lo = (int)ceilf(fmaxf((gy - ey - 3.5f) * 0.25f, 0.f));
    const int r_hi = (int)floorf(fminf((gy + ey - 0.5f) * 0.25f, (float)(SPR - 1)));
    const float det = fmaf(a, c, -b * b);
    const float aq = a * qm;
    const float ra = rcp_approx(a);
    const float dys = b * sqrt_approx(qm * rdet * rcp_approx(c));
    MaskT mask = 0;
    for (int r = r_lo; r <= r_hi; ++r) {
        const float u0 = fmaxf((float)(4 * r) + 0.5f - gy, -ey);
        const float u1 = fminf((float)(4 * r) + 3.5f - gy, ey);
        const float dl = fminf(fmaxf(dys, u0), u1);
        const float dr = fminf(fmaxf(-dys, u0), u1);
        const float sl = sqrt_approx(fmaxf(0.f, fmaf(-det, dl * dl, aq)));
        const float sr = sqrt_approx(fmaxf(0.f, fmaf(-det, dr * dr, aq)));
        const float xl = gx - fmaf(b, dl, sl) * ra - xmargin;
        const float xh = gx + fmaf(-b, dr, sr) * ra + xmargin;
        mask |= MaskT(span_bits<SPR>(xl, xh)) << (r * SPR);
    }
    return mask;
}

// Builds the staged record of one splat and the mask of the sub-blocks that
// its opacity-aware ellipse (§3.4) q = a dx^2 + 2 b dx dy + c dy^2 <= qc
// reaches: with ELLIPSE the sub-blocks that the ellipse itself meets
// (ellipse_subblock_mask), else those that its bounding box meets (half-
// widths sqrt(qc Sigma'_xx), sqrt(qc Sigma'_yy) with Sigma' = [[c, -b],
// [-b, a]] / det). The ellipse is grown to qm = 1.001 qc + 1e-3 and the
// ranges by a relative and an absolute margin, well above the error of the
// approximate reciprocal and square roots, so no pixel inside the exact
// ellipse is left out; a sub-block visited without need adds w = 0. The
// ellipse's mask costs more arithmetic per staged splat and saves visits
// (13 % of them on the 1080p / 1M frame): a gain where a visit is dear (the
// backward), not in the forward. WS_CFG_BOX_MASKS takes the box's mask
// everywhere; the results are the same bits either way.
template <typename G, bool ELLIPSE, typename Splats>
__device__ __forceinline__ void stage_splat(const Frame& f, float ox, float oy, const Splats& sp, uint32_t g,
                                            SplatRec* dst, typename G::Mask& mask) {
    float a, b, c, op, gx, gy;
    float4 col;
    sp.load(g, ox, oy, gx, gy, a, b, c, op, col);
    const float L = lg2_approx(op);
    // the record first: its registers are free before the mask's arithmetic
    float ct = 0.f, st = 0.f;
    if (ELLIPSE) axis_basis(col.w, ct, st);
    dst->geo = make_float4(-gx, -gy, -0.5f * kLog2e * a, -kLog2e * b);
    dst->geo2 = make_float4(-0.5f * kLog2e * c, L, ct, st);
    dst->col = make_float4(col.x, col.y, col.z, 0.f);
    const float qc = (f.flags & WS_CFG_FIXED_RADIUS) ? 2.f * kLn255 : fmaxf(0.f, kTwoLn2 * (L - kLog2AlphaMin));
    const float qm = fmaf(qc, 1.001f, 1e-3f);
    const float rdet = rcp_approx(fmaf(a, c, -b * b));
    const float ex = sqrt_approx(qm * c * rdet) * 1.0001f + 1e-3f;
    const float ey = sqrt_approx(qm * a * rdet) * 1.0001f + 1e-3f;
    using M = typename G::Mask;
    if (ELLIPSE && !(f.flags & WS_CFG_BOX_MASKS))
        mask = ellipse_subblock_mask<G::SPR, M>(gx, gy, a, b, c, qm, rdet, ey, fmaf(ex, 1e-4f, 1e-3f));
    else
        mask = box_subblock_mask<G::SPR, M>(gx - ex, gx + ex, gy - ey, gy + ey);
}

// e of splat_log2_alpha for a pair of pixels of one column: the same
// operations in the same order, so the same bits.
__device__ __forceinline__ F2 splat_log2_alpha2(float dx, F2 dy, const float4& geo, const float4& geo2) {
    const F2 u = fma2(dup2(geo.z), dup2(dx), mul2(dup2(geo.w), dy));
    return fma2(dup2(dx), u, fma2(mul2(dup2(geo2.x), dy), dy, dup2(geo2.y)));
}

// Forward state of a thread's pixels: front to back, C += c a T, T -= a T.
template <typename G, int PX>
struct FwdPixels {
    static constexpr int NP = PX / 2;
    int ix, iy0;
    float px;
    F2 py[NP], T[NP], C0[NP], C1[NP], C2[NP];
    uint32_t last[PX];

    __device__ __forceinline__ void init(int warp, int lane) {
        G::pixel(warp, lane, ix, iy0);
        px = (float)ix + 0.5f;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const float y = (float)(iy0 + 2 * p) + 0.5f;
            py[p] = pack2(y, y + 1.f);
            T[p] = dup2(1.f);
            C0[p] = C1[p] = C2[p] = dup2(0.f);
            last[2 * p] = last[2 * p + 1] = 0;
        }
    }

    // Composites the visits of this lane's stream (`row`, `steps` entries,
    // the null splat past its own). rel0: the 1-based list position of
    // staged index 0. A null visit and one below the 1/255 test add w = 0,
    // which leaves C and T bit for bit unchanged, so per pixel the
    // compositing order and arithmetic are those of a plain front-to-back
    // loop. The last composited index is kept 1-based and made a list
    // position once at the end.
    __device__ __forceinline__ void walk(const SplatRec* s_rec, const uint8_t* row, int steps, uint32_t rel0) {
        int lastk[PX];
#pragma unroll
        for (int k = 0; k < PX; ++k) lastk[k] = 0;
        int j = row[0];
#pragma unroll 4
        for (int it = 0; it < steps; ++it) {
            const SplatRec& r = s_rec[j];
            const int j1 = j + 1;
            j = row[it + 1];  // the next entry's latency overlaps this visit
            const float4 geo = r.geo;
            const float2 g2 = *reinterpret_cast<const float2*>(&r.geo2);
            const float4 geo2 = make_float4(g2.x, g2.y, 0.f, 0.f);
            const float4 col = r.col;
            const float dx = __fadd_rn(px, geo.x);
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const F2 e2 = splat_log2_alpha2(dx, add2(py[p], dup2(geo.y)), geo, geo2);
                float e[2], al[2];
                unpack2(e2, e[0], e[1]);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const bool keep = e[h] >= kLog2AlphaMin;
                    const float alpha = fminf(kAlphaMax, ex2_approx(e[h]));
                    al[h] = keep ? alpha : 0.f;
                    lastk[2 * p + h] = keep ? j1 : lastk[2 * p + h];
                }
                const F2 w = mul2(pack2(al[0], al[1]), T[p]);
                C0[p] = fma2(dup2(col.x), w, C0[p]);
                C1[p] = fma2(dup2(col.y), w, C1[p]);
                C2[p] = fma2(dup2(col.z), w, C2[p]);
                T[p] = fma2(w, dup2(-1.f), T[p]);  // T - w
            }
        }
#pragma unroll
        for (int k = 0; k < PX; ++k)
            if (lastk[k]) last[k] = rel0 + (uint32_t)(lastk[k] - 1);
    }
};

// Splats the backward stages at a time, the visits (a staged splat and a
// sub-block that it reaches) whose rows it holds at a time, and the
// granularity of the splat spans it processes: a span of vis_unit splats
// always fits. At 16-pixel tiles 96 and 128: 31 KB, six blocks of which leave
// the L1 56 KB of the SM's 256. 128 splats (35 KB a block) shrink it to 23 KB
// and took the 64-view backward from 20.6 to 23.1 ms; 64 splats end their
// spans early (22.5 ms), and rows for 64 visits double the barriers (21.9).
template <int TS>
__host__ __device__ constexpr int bwd_batch() { return TS == 16 ? 96 : 64; }
template <int TS>
__host__ __device__ constexpr int vis_cap() { return TS == 8 ? 32 : 128; }
template <int TS>
__host__ __device__ constexpr int vis_unit() { return TS == 32 ? 2 : 8; }

// The pair records of a backward: partials 0..7 of slot s at p8[2 s], p8[2 s
// + 1] (one 32-byte sector), partial 8 at p9[s].
struct PairRecords {
    float4* p8;
    float* p9;
};

// The pair records in a backward's scratch: 36 bytes per key of capacity,
// the 32-byte parts first.
inline PairRecords pair_records(void* scratch, int64_t key_capacity) {
    float4* p8 = static_cast<float4*>(scratch);
    return {p8, reinterpret_cast<float*>(p8 + 2 * (size_t)key_capacity)};
}

// Shared memory of the backward, staging BATCH splats.
template <int TS, int PX, int BATCH>
struct BwdSmem {
    using G = TileGeom<TS, PX>;
    static constexpr int VCAP = vis_cap<TS>();
    static constexpr int ROW = BATCH + 16;  // entries of a visit list
    SplatRec rec[BATCH + 1];
    // row v: the 16 pixels' (w, dp) of visit v, a float4 (w, w, dp, dp) for
    // each vertical pair of pixels, and 16 bytes of padding (a thread per row
    // then reads its float4s without bank conflicts); row VCAP takes the null
    // visits
    float4 vrow[(VCAP + 1) * 9];
    __align__(16) uint16_t list[G::NSB * ROW];  // staged index | visit << 8
    // dL/dC of each sub-block's pixels: 8 pairs (r, r, g, g), 8 pairs (b, b),
    // in rows of 52 floats, whose float4s fall in distinct banks for eight
    // neighbouring sub-blocks (rows of 48 cost the 64-view step 25 %)
    __align__(16) float dC[G::NSB][52];
    typename G::Mask mask[BATCH];
    uint32_t slot[BATCH];
    uint16_t vis[VCAP];        // staged index | sub-block << 8
    uint16_t base[BATCH + 2];  // visits of the staged splats before each
};

// Backward state of a thread's pixels, walked back to front from the final
// transmittance. With b = the colour behind the splat, normalised by the
// transmittance after it and projected on the pixel's dL/dC (b starts as
// bg . dL/dC, b <- a s + (1 - a) b with s = c . dL/dC):
//   dL/dc = w dL/dC with w = a T,   dL/da = T (s - b),
// and, unless the alpha was clamped at 0.99, sigma dL/dsigma = dL/dpower =
// a dL/da =: dp (a = sigma G there) with power = -1/2 d^T Q d, giving
// d/dmean = Q d dp and the conic's derivatives from dp u^2, dp u v, dp v^2
// in the splat's axis basis. So w and dp are all a visit's pixels contribute:
// the walk, which must follow the list, stores the two per pixel, and the
// sums over the sub-block's 16 pixels are taken afterwards by one thread per
// visit, with no shuffle and every lane busy.
template <int TS, int PX>
struct BwdPixels {
    using G = TileGeom<TS, PX>;
    static constexpr int NP = PX / 2;
    float px;
    F2 py[NP], T[NP], b[NP], dC[NP][3];

    // ix, iy0: this lane's pixels (TileGeom::pixel); tf, bf, dc: the
    // transmittance and b behind the span walked (the whole list's: t_final
    // and bg . dL/dC) and dL/dC, zeros outside the image; inside: pixels past
    // the image's edge have no position (NaN), so that nothing composites
    // there. s_dC: this lane's sub-block's row of BwdSmem::dC.
    __device__ __forceinline__ void init(int lane, int ix, int iy0, const bool (&inside)[PX], const float (&tf)[PX],
                                         const float (&bf)[PX], const float (&dc)[PX][3], float* s_dC) {
        px = (float)ix + 0.5f;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const float y = (float)(iy0 + 2 * p) + 0.5f;
            py[p] = pack2(inside[2 * p] ? y : NAN, inside[2 * p + 1] ? y + 1.f : NAN);
            T[p] = pack2(tf[2 * p], tf[2 * p + 1]);
#pragma unroll
            for (int c = 0; c < 3; ++c) dC[p][c] = pack2(dc[2 * p][c], dc[2 * p + 1][c]);
            b[p] = pack2(bf[2 * p], bf[2 * p + 1]);
            const int k = p * 4 + lane % G::LPS;  // pair of pixels: row pair * 4 + column
            *reinterpret_cast<float4*>(s_dC + 4 * k) =
                make_float4(dc[2 * p][0], dc[2 * p + 1][0], dc[2 * p][1], dc[2 * p + 1][1]);
            *reinterpret_cast<float2*>(s_dC + 32 + 2 * k) = make_float2(dc[2 * p][2], dc[2 * p + 1][2]);
        }
    }

    // A visit of this lane's stream: advances the pixels' state and stores
    // their (w, dp) in the visit's row. A pixel that does not composite the
    // splat has alpha = 0, which makes its w and dp zero and leaves T and b
    // as they are, unless a factor is infinite or NaN: a colour, dL/dC, what
    // lies behind (the background, the segments behind this one) or a product
    // of them that overflows. FINITE = false, taken where any of them is not
    // walkable, selects instead of multiplying, so that such a value reaches
    // only the pixels and splats that it belongs to.
    template <bool FINITE>
    __device__ __forceinline__ void visit(const float4& geo, const float2& g2, const float4& col, float4* row) {
        const float4 geo2 = make_float4(g2.x, g2.y, 0.f, 0.f);
        const float dx = __fadd_rn(px, geo.x);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const F2 e2 = splat_log2_alpha2(dx, add2(py[p], dup2(geo.y)), geo, geo2);
            float e[2], al[2], rt[2], au[2];
            unpack2(e2, e[0], e[1]);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float raw = e[h] >= kLog2AlphaMin ? ex2_approx(e[h]) : 0.f;
                al[h] = fminf(kAlphaMax, raw);
                au[h] = raw < kAlphaMax ? raw : 0.f;        // no gradient through the clamp
                rt[h] = rcp_approx(__fsub_rn(1.f, al[h]));  // 1 for alpha = 0: T unchanged
            }
            const F2 alpha = pack2(al[0], al[1]);
            T[p] = mul2(T[p], pack2(rt[0], rt[1]));
            const F2 sc = fma2(dup2(col.z), dC[p][2], fma2(dup2(col.y), dC[p][1], mul2(dup2(col.x), dC[p][0])));
            const F2 d = fma2(b[p], dup2(-1.f), sc);  // s - b
            const F2 w = mul2(alpha, T[p]);
            const F2 dp = mul2(pack2(au[0], au[1]), mul2(d, T[p]));
            const F2 bn = fma2(alpha, d, b[p]);
            float4 o;
            unpack2(w, o.x, o.y);
            unpack2(dp, o.z, o.w);
            if (FINITE) {
                b[p] = bn;
            } else {
                float b0, b1, n0, n1;
                unpack2(b[p], b0, b1);
                unpack2(bn, n0, n1);
                b[p] = pack2(al[0] > 0.f ? n0 : b0, al[1] > 0.f ? n1 : b1);
                o.x = al[0] > 0.f ? o.x : 0.f;
                o.y = al[1] > 0.f ? o.y : 0.f;
                o.z = au[0] > 0.f ? o.z : 0.f;
                o.w = au[1] > 0.f ? o.w : 0.f;
            }
            row[p * 4] = o;
        }
    }

    // One thread's sum over the 16 pixels of a visit of splat r in sub-block
    // sb, in a fixed order, written over the visit's row: dp Q d (x, y) and
    // dp (u^2, u v, v^2), dp, w dL/dC, without the constant factors that
    // batch() applies once per splat.
    template <bool FINITE>
    __device__ static __forceinline__ void sum_visit(const SplatRec& r, int sb, const float* s_dC, float4* row) {
        const float4 geo = r.geo, geo2 = r.geo2;
        const float x0 = (float)((sb % G::SPR) * 4) + 0.5f, y0 = (float)((sb / G::SPR) * 4) + 0.5f;
        const F2 st = dup2(geo2.w), ct = dup2(geo2.z), zero = dup2(0.f);
        bool any = FINITE;
        F2 S0 = zero, Sx = zero, Sy = zero, Suu = zero, Suv = zero, Svv = zero, Cr = zero, Cg = zero, Cb = zero;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float dx = __fadd_rn(x0 + (float)(k & 3), geo.x);
            const float y = y0 + (float)(2 * (k >> 2));
            const F2 dy = add2(pack2(y, y + 1.f), dup2(geo.y));
            const F2 u = fma2(st, dy, dup2(__fmul_rn(geo2.z, dx))), v = fma2(ct, dy, dup2(__fmul_rn(-geo2.w, dx)));
            const float4 q = row[k];
            const F2 w = pack2(q.x, q.y), dp = pack2(q.z, q.w);
            const F2 du = mul2(dp, u), dv = mul2(dp, v);
            float4 rg = *reinterpret_cast<const float4*>(s_dC + 4 * k);
            float2 bb = *reinterpret_cast<const float2*>(s_dC + 32 + 2 * k);
            if (!FINITE) {  // only the pixels that composite the splat
                any = any || q.x != 0.f || q.y != 0.f || q.z != 0.f || q.w != 0.f;
                if (q.x == 0.f) rg.x = rg.z = bb.x = 0.f;
                if (q.y == 0.f) rg.y = rg.w = bb.y = 0.f;
            }
            S0 = add2(S0, dp);
            Sx = fma2(dp, dup2(dx), Sx);
            Sy = fma2(dp, dy, Sy);
            Suu = fma2(du, u, Suu);
            Suv = fma2(du, v, Suv);
            Svv = fma2(dv, v, Svv);
            Cr = fma2(w, pack2(rg.x, rg.y), Cr);
            Cg = fma2(w, pack2(rg.z, rg.w), Cg);
            Cb = fma2(w, pack2(bb.x, bb.y), Cb);
        }
        const float sx = sum2(Sx), sy = sum2(Sy), hb = __fmul_rn(0.5f, geo.w);
        row[0] = make_float4(__fmaf_rn(geo.z, sx, __fmul_rn(hb, sy)), __fmaf_rn(geo2.x, sy, __fmul_rn(hb, sx)),
                             sum2(Suu), sum2(Suv));
        row[1] = make_float4(sum2(Svv), sum2(S0), sum2(Cr), sum2(Cg));
        row[2].x = sum2(Cb);
        if (!any) row[0] = row[1] = row[2] = make_float4(0.f, 0.f, 0.f, 0.f);
    }

    // The visit lists of this warp's streams over the staged splats [lo, hi),
    // back to front (as build_lists), each entry with the visit's row; also
    // vis[]. Returns the longest list's length.
    template <int BATCH>
    __device__ __forceinline__ int build_visits(BwdSmem<TS, PX, BATCH>& sm, int lo, int hi, int vis0, int warp,
                                                int lane) {
        using S = BwdSmem<TS, PX, BATCH>;
        static_assert(BATCH < 256 && S::VCAP < 256 && S::ROW % 8 == 0, "8-bit indices and visits, 16-byte rows");
        uint16_t* rows = sm.list + warp * G::SPW * S::ROW;
        constexpr uint32_t kNull2 = 0x00010001u * (uint32_t)(BATCH | (S::VCAP << 8));
        uint4* mine = reinterpret_cast<uint4*>(rows + (lane / G::LPS) * S::ROW);
        for (int v = lane % G::LPS; v <= (hi - lo + 1) >> 3; v += G::LPS) mine[v] = make_uint4(kNull2, kNull2, kNull2, kNull2);
        __syncwarp();
        const uint32_t lt = lanemask_lt();
        const int sb0 = warp * G::SPW;
        int c[G::SPW];
#pragma unroll
        for (int t = 0; t < G::SPW; ++t) c[t] = 0;
        for (int k = 0; k < hi - lo; k += 32) {
            const bool in = k + lane < hi - lo;
            const int j = hi - 1 - k - lane;
            const typename G::Mask full = in ? sm.mask[j] : typename G::Mask(0);
            const uint32_t m = (uint32_t)(full >> sb0);
            int v = in ? (int)sm.base[j] - vis0 + popc_mask(full & ((typename G::Mask(1) << sb0) - 1)) : 0;
#pragma unroll
            for (int t = 0; t < G::SPW; ++t) {
                const bool bit = (m >> t) & 1u;
                const uint32_t bal = __ballot_sync(kFull, bit);
                if (bit) {
                    rows[t * S::ROW + c[t] + __popc(bal & lt)] = (uint16_t)(j | (v << 8));
                    sm.vis[v] = (uint16_t)(j | ((sb0 + t) << 8));
                    ++v;
                }
                c[t] += __popc(bal);
            }
        }
        __syncwarp();
        int steps = 0;
#pragma unroll
        for (int t = 0; t < G::SPW; ++t) steps = max(steps, c[t]);
        return steps;
    }

    // This lane's visits of one span. The next visit's record is loaded
    // before this one's stores (which the compiler must assume to alias it),
    // the entry after it before that, so their latencies overlap the
    // arithmetic: 157 -> 152 us on the 720p backward call.
    template <bool FINITE, typename S>
    __device__ __forceinline__ void walk(const S& sm, const uint16_t* row, float4* vrow, int steps) {
        uint32_t code = row[0], next = row[1];
        const SplatRec* r = sm.rec + (code & 255u);
        float4 geo = r->geo, col = r->col;
        float2 g2 = *reinterpret_cast<const float2*>(&r->geo2);
#pragma unroll FINITE ? 4 : 1
        for (int it = 0; it < steps; ++it) {
            const float4 geo0 = geo, col0 = col;
            const float2 g20 = g2;
            float4* dst = vrow + (code >> 8) * 9;
            code = next;
            next = row[it + 2];
            r = sm.rec + (code & 255u);
            geo = r->geo;
            col = r->col;
            g2 = *reinterpret_cast<const float2*>(&r->geo2);
            visit<FINITE>(geo0, g20, col0, dst);
        }
    }

    // Walks the staged splats [0, cnt) back to front. The splats are taken
    // in spans of at most vis_cap visits: every stream walks its visits of
    // the span (visit), one thread per visit sums its pixels (sum_visit),
    // and one thread per splat adds its visits (contiguous, its sub-blocks
    // ascending) and writes its record at the pair's emission slot. Which
    // visits exist is known from the masks, so nothing is cleared or
    // flagged.
    template <bool FINITE, int BATCH>
    __device__ __forceinline__ void batch(BwdSmem<TS, PX, BATCH>& sm, int cnt, int warp, int lane,
                                          const PairRecords& out) {
        using S = BwdSmem<TS, PX, BATCH>;
        if (warp == 0) {  // exclusive scan of the visit counts
            uint32_t run = 0;
            for (int k = 0; k < cnt; k += 32) {
                const uint32_t n = k + lane < cnt ? (uint32_t)popc_mask(sm.mask[k + lane]) : 0u;
                uint32_t x = n;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(kFull, x, o);
                    if (lane >= o) x += y;
                }
                if (k + lane < cnt) sm.base[k + lane] = (uint16_t)(run + x - n);
                run += __shfl_sync(kFull, x, 31);
            }
            if (lane == 0) sm.base[cnt] = (uint16_t)run;
        }
        __syncthreads();
        const uint16_t* row = sm.list + (warp * G::SPW + lane / G::LPS) * S::ROW;
        float4* vrow = sm.vrow + lane % G::LPS;
        constexpr int U = vis_unit<TS>();
        for (int hi = cnt; hi > 0;) {
            // the longest span [lo, hi), lo a multiple of U, that fits
            int lo = ((hi - 1) / U - lane) * U;
            const int end = sm.base[hi];
            const bool fits = lo >= 0 && end - (int)sm.base[max(lo, 0)] <= S::VCAP;
            lo = ((hi - 1) / U - (__popc(__ballot_sync(kFull, fits)) - 1)) * U;
            const int vis0 = sm.base[lo];
            const int steps = build_visits<BATCH>(sm, lo, hi, vis0, warp, lane);
            walk<FINITE>(sm, row, vrow, steps);
            __syncthreads();
            for (int v = threadIdx.x; v < end - vis0; v += G::THREADS) {
                const uint32_t c = sm.vis[v];
                sum_visit<FINITE>(sm.rec[c & 255u], (int)(c >> 8), sm.dC[c >> 8], sm.vrow + v * 9);
            }
            __syncthreads();
            for (int j = lo + threadIdx.x; j < hi; j += G::THREADS) {
                float4 a = make_float4(0.f, 0.f, 0.f, 0.f), c = a;
                float d = 0.f;
                const int v1 = (int)sm.base[j + 1] - vis0;
                for (int v = (int)sm.base[j] - vis0; v < v1; ++v) {
                    const float4 x = sm.vrow[v * 9], y = sm.vrow[v * 9 + 1];
                    a.x += x.x;
                    a.y += x.y;
                    a.z += x.z;
                    a.w += x.w;
                    c.x += y.x;
                    c.y += y.y;
                    c.z += y.z;
                    c.w += y.w;
                    d += sm.vrow[v * 9 + 2].x;
                }
                const size_t s = sm.slot[j];
                out.p8[2 * s] = make_float4(-2.f * kLn2 * a.x, -2.f * kLn2 * a.y, -0.5f * a.z, -a.w);
                out.p8[2 * s + 1] = make_float4(-0.5f * c.x, c.y, c.z, c.w);
                out.p9[s] = d;
            }
            __syncthreads();
            hi = lo;
        }
    }
    __device__ static __forceinline__ int popc_mask(uint32_t m) { return __popc(m); }
    __device__ static __forceinline__ int popc_mask(unsigned long long m) { return __popcll(m); }
};

// Tile of a frame that the backward's launch index b takes: the tile rows
// centre-out (c, c + 1, c - 1, c + 2, ..., c = (TY - 1) / 2, a bijection onto
// [0, TY) for either parity of TY), each row left to right. The rows near
// the image's centre, where the lists are longest in views of a centred
// scene, start first and the short border rows fill the end of the launch;
// neighbouring launches stay neighbouring tiles. Each tile's computation is
// the same whatever the order.
__device__ __forceinline__ int centre_out_tile(const Frame& f, int b) {
    const int r = b / f.TX, tx = b - r * f.TX;
    const int c = (f.TY - 1) / 2;
    const int ty = (r & 1) ? c + (r + 1) / 2 : c - r / 2;
    return ty * f.TX + tx;
}

// Emission slot of the pair (tile (tx, ty), Gaussian g): its first slot
// slot_of(g) plus the tile's row-major rank in g's rectangle.
template <typename SlotBase>
__device__ __forceinline__ uint32_t pair_slot(SlotBase slot_of, const uint2* __restrict__ rect, uint32_t g, int tx,
                                              int ty) {
    const uint2 rc = __ldg(rect + g);
    const uint32_t x0 = rc.x & 0xffffu, y0 = rc.x >> 16, x1 = rc.y & 0xffffu;
    return slot_of(g) + (ty - y0) * (x1 - x0 + 1) + (tx - x0);
}

// Slot-ordered sum of a Gaussian's nrec pair records (slots first ..) into
// pr: the loads of four records are issued before their adds, and the adds
// keep slot order (a record past nrec adds +0, which leaves a sum that
// started at +0 bit for bit unchanged), so the result is that of the plain
// loop with a quarter of its dependent load latencies.
__device__ __forceinline__ void sum_pair_records(const float4* __restrict__ p8, const float* __restrict__ p9,
                                                 size_t first, uint32_t nrec, float (&pr)[kPart]) {
    for (uint32_t s = 0; s < nrec; s += 4) {
        float4 a[4], b[4];
        float c[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const bool ok = s + k < nrec;
            const size_t t = first + s + k;
            a[k] = ok ? __ldg(p8 + 2 * t) : make_float4(0.f, 0.f, 0.f, 0.f);
            b[k] = ok ? __ldg(p8 + 2 * t + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
            c[k] = ok ? __ldg(p9 + t) : 0.f;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            pr[0] += a[k].x;
            pr[1] += a[k].y;
            pr[2] += a[k].z;
            pr[3] += a[k].w;
            pr[4] += b[k].x;
            pr[5] += b[k].y;
            pr[6] += b[k].z;
            pr[7] += b[k].w;
            pr[8] += c[k];
        }
    }
}

// Stages list positions [start, start + cnt) of a tile: records and masks,
// and (WITH_SLOT) each pair's emission slot. The staging of the backward
// (WITH_SLOT) builds the ellipse's sub-block
// masks, the forward's the bounding box's. g0: vals[start + threadIdx.x], which
// the caller has loaded. Returns whether the records that this thread staged
// are walkable (WITH_SLOT).
template <typename G, bool WITH_SLOT, typename Splats, typename SlotBase>
__device__ __forceinline__ bool stage_batch(const Frame& f, float ox, float oy, int tx, int ty, uint32_t start,
                                            int cnt, uint32_t g0, const uint32_t* __restrict__ vals,
                                            const Splats& sp, const uint2* __restrict__ rect, SlotBase slot_of,
                                            SplatRec* s_rec, typename G::Mask* s_mask, uint32_t* s_slot) {
    bool ok = true;
    for (int j = threadIdx.x; j < cnt; j += G::THREADS) {
        const uint32_t g = j == (int)threadIdx.x ? g0 : __ldg(vals + start + j);
        typename G::Mask m;
        stage_splat<G, WITH_SLOT>(f, ox, oy, sp, g, s_rec + j, m);
        s_mask[j] = m;
        if (WITH_SLOT) {
            s_slot[j] = pair_slot(slot_of, rect, g, tx, ty);
            const SplatRec& r = s_rec[j];
            // one sum of magnitudes: eleven comparisons took 1 % of a step of short lists
            const float geo = fabsf(r.geo.x) + fabsf(r.geo.y) + fabsf(r.geo.z) + fabsf(r.geo.w);
            const float geo2 = fabsf(r.geo2.x) + fabsf(r.geo2.y) + fabsf(r.geo2.z) + fabsf(r.geo2.w);
            ok = ok && walkable(geo + geo2 + (fabsf(r.col.x) + fabsf(r.col.y) + fabsf(r.col.z)));
        }
    }
    return ok;
}

// vals[start + threadIdx.x] for the threads that stage it of a batch of the list
// [.., end), loaded a batch ahead: the records' addresses are then known when
// their turn comes.
template <typename G, int BATCH>
__device__ __forceinline__ uint32_t first_value(const uint32_t* __restrict__ vals, uint32_t start, uint32_t end) {
    return threadIdx.x < BATCH && start + threadIdx.x < end ? __ldg(vals + start + threadIdx.x) : 0u;
}

struct NoSlot {
    __device__ __forceinline__ uint32_t operator()(uint32_t) const { return 0u; }
};

// Forward of one tile: stages the list a batch at a time, and each warp
// builds its streams' visit lists and composites them (FwdPixels::walk);
// then writes image = C + T bg, the final transmittance and the 1-based list
// position of the last composited splat.
template <int TS, int PX, typename Splats>
__device__ __forceinline__ void blend_tile(const Frame& f, int tile, uint2 range, const uint32_t* __restrict__ vals,
                                           const Splats& sp, float* __restrict__ image, float* __restrict__ t_final,
                                           uint32_t* __restrict__ n_contrib) {
    using G = TileGeom<TS, PX>;
    constexpr int BATCH = fwd_batch<TS>();
    __shared__ SplatRec s_rec[BATCH + 1];
    __shared__ typename G::Mask s_mask[BATCH];
    __shared__ __align__(16) uint8_t s_list[G::NSB * list_row<BATCH>()];
    const int tx = tile % f.TX, ty = tile / f.TX;
    const float ox = (float)(tx * TS), oy = (float)(ty * TS);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint8_t* rows = s_list + warp * G::SPW * list_row<BATCH>();
    init_null_splat(s_rec, BATCH);
    FwdPixels<G, PX> P;
    P.init(warp, lane);
    uint32_t g0 = first_value<G, BATCH>(vals, range.x, range.y);
    for (uint32_t start = range.x; start < range.y; start += BATCH) {
        const int cnt = (int)min((uint32_t)BATCH, range.y - start);
        __syncthreads();
        stage_batch<G, false>(f, ox, oy, tx, ty, start, cnt, g0, vals, sp, nullptr, NoSlot{}, s_rec, s_mask, nullptr);
        g0 = first_value<G, BATCH>(vals, start + BATCH, range.y);
        __syncthreads();
        const int steps = build_lists<G, BATCH, false>(s_mask, 0, cnt, rows, warp, lane);
        P.walk(s_rec, rows + (lane / G::LPS) * list_row<BATCH>(), steps, start + 1 - range.x);
    }
    const int gx = tx * TS + P.ix;
#pragma unroll
    for (int k = 0; k < PX; ++k) {
        const int gy = ty * TS + P.iy0 + k;
        if (gx < f.W && gy < f.H) {
            const size_t pix = (size_t)gy * f.W + gx;
            float c[2][4];
            unpack2(P.T[k / 2], c[0][3], c[1][3]);
            unpack2(P.C0[k / 2], c[0][0], c[1][0]);
            unpack2(P.C1[k / 2], c[0][1], c[1][1]);
            unpack2(P.C2[k / 2], c[0][2], c[1][2]);
            const float(&o)[4] = c[k & 1];
            image[3 * pix] = fmaf(o[3], f.bg[0], o[0]);
            image[3 * pix + 1] = fmaf(o[3], f.bg[1], o[1]);
            image[3 * pix + 2] = fmaf(o[3], f.bg[2], o[2]);
            t_final[pix] = o[3];
            n_contrib[pix] = P.last[k];
        }
    }
}

// dL/dC of this lane's pixels, zeros outside the image: d_image, or in an L2
// training step d_image - target with the image in d_image's place. Returns
// whether they are walkable.
template <int PX>
__device__ __forceinline__ bool load_dc(const Frame& f, int gx, int gy0, const float* __restrict__ d_image,
                                        const float* __restrict__ target, float (&dc)[PX][3]) {
    bool ok = true;
#pragma unroll
    for (int k = 0; k < PX; ++k) {
        const int gy = gy0 + k;
        const bool inside = gx < f.W && gy < f.H;
        const size_t pix = inside ? (size_t)gy * f.W + gx : 0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float g = inside ? d_image[3 * pix + c] : 0.f;
            dc[k][c] = target && inside ? g - __ldg(target + 3 * pix + c) : g;
            ok = ok && walkable(dc[k][c]);
        }
    }
    return ok;
}

__device__ __forceinline__ float dot3(const float* a, const float (&d)[3]) {
    return fmaf(a[2], d[2], fmaf(a[1], d[1], a[0] * d[0]));
}

// Long lists are cut into segments that the backward walks at the same time
// (launch_tile_order): one tile of the 6-view step has 4,819 of its 1.9M
// pairs, and its walk alone, about 100 ns a splat, took as long as all
// others together. segment_state finds, for one segment, what the segments in
// front of it have to know: its transmittance T (from 1 at its front) and its
// colour D, composited from T = 1 and projected on dL/dC. Segment k then starts
// from T = T_0 ... T_k and b = D_{k+1} + T_{k+1} (D_{k+2} + ... T_last bg . dL/dC):
// sums of non-negative weights, nothing subtracted.
template <int TS, int PX>
__device__ __forceinline__ void segment_state(const Frame& f, int tile, uint32_t first, uint32_t last,
                                              const uint32_t* __restrict__ vals, const float4* __restrict__ splats,
                                              const float* __restrict__ d_image, const float* __restrict__ target,
                                              float2* __restrict__ state) {
    using G = TileGeom<TS, PX>;
    constexpr int BATCH = fwd_batch<TS>();
    constexpr int NP = PX / 2;
    __shared__ SplatRec s_rec[BATCH + 1];
    __shared__ typename G::Mask s_mask[BATCH];
    __shared__ __align__(16) uint8_t s_list[G::NSB * list_row<BATCH>()];
    const int tx = tile % f.TX, ty = tile / f.TX;
    const float ox = (float)(tx * TS), oy = (float)(ty * TS);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint8_t* rows = s_list + warp * G::SPW * list_row<BATCH>();
    const uint8_t* row = rows + (lane / G::LPS) * list_row<BATCH>();
    const FloatSplats sp{splats};
    init_null_splat(s_rec, BATCH);
    int ix, iy0;
    G::pixel(warp, lane, ix, iy0);
    float dc[PX][3];
    load_dc<PX>(f, tx * TS + ix, ty * TS + iy0, d_image, target, dc);
    const float px = (float)ix + 0.5f;
    F2 py[NP], T[NP];
    float D[PX];
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        const int gy = ty * TS + iy0 + 2 * p;  // (pixels past the image's edge have no position)
        const float y = (float)(iy0 + 2 * p) + 0.5f;
        const bool col_in = tx * TS + ix < f.W;
        py[p] = pack2(col_in && gy < f.H ? y : NAN, col_in && gy + 1 < f.H ? y + 1.f : NAN);
        T[p] = dup2(1.f);
        D[2 * p] = D[2 * p + 1] = 0.f;
    }
    uint32_t g0 = first_value<G, BATCH>(vals, first, last);
    for (uint32_t start = first; start < last; start += BATCH) {
        const int cnt = (int)min((uint32_t)BATCH, last - start);
        __syncthreads();
        stage_batch<G, false>(f, ox, oy, tx, ty, start, cnt, g0, vals, sp, nullptr, NoSlot{}, s_rec, s_mask, nullptr);
        g0 = first_value<G, BATCH>(vals, start + BATCH, last);
        __syncthreads();
        const int steps = build_lists<G, BATCH, false>(s_mask, 0, cnt, rows, warp, lane);
        int j = row[0];
#pragma unroll 4
        for (int it = 0; it < steps; ++it) {
            const SplatRec& r = s_rec[j];
            j = row[it + 1];
            const float4 geo = r.geo, col = r.col;
            const float2 g2 = *reinterpret_cast<const float2*>(&r.geo2);
            const float4 geo2 = make_float4(g2.x, g2.y, 0.f, 0.f);
            const float dx = __fadd_rn(px, geo.x);
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const F2 e2 = splat_log2_alpha2(dx, add2(py[p], dup2(geo.y)), geo, geo2);
                float e[2], w[2];
                unpack2(e2, e[0], e[1]);
                F2 al = pack2(e[0] >= kLog2AlphaMin ? fminf(kAlphaMax, ex2_approx(e[0])) : 0.f,
                              e[1] >= kLog2AlphaMin ? fminf(kAlphaMax, ex2_approx(e[1])) : 0.f);
                al = mul2(al, T[p]);
                T[p] = fma2(al, dup2(-1.f), T[p]);
                unpack2(al, w[0], w[1]);
                const float cc[3] = {col.x, col.y, col.z};
#pragma unroll
                for (int h = 0; h < 2; ++h)  // (an infinite colour stays with its pixels)
                    if (e[h] >= kLog2AlphaMin) D[2 * p + h] = fmaf(w[h], dot3(cc, dc[2 * p + h]), D[2 * p + h]);
            }
        }
    }
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        float t0, t1;
        unpack2(T[p], t0, t1);
        state[(size_t)threadIdx.x * PX + 2 * p] = make_float2(t0, D[2 * p]);
        state[(size_t)threadIdx.x * PX + 2 * p + 1] = make_float2(t1, D[2 * p + 1]);
    }
}

// The part of a tile's list that a backward block walks: positions [lo, hi)
// of the list; states (null for a whole list): the segment states of the
// tile's nseg segments, of which this is number seg.
struct BwdSpan {
    uint32_t lo, hi;
    const float2* states;
    uint32_t seg, nseg;
};

// Backward of (a span of) one tile from the stored final transmittance: each
// pair's 9 partials at its emission slot (see BwdPixels). offsets[g]: the first
// emission slot of Gaussian g's pairs (in a batch, of this view's). d_image and
// target: load_dc. FINITE = true stops and returns false when a staged record,
// a dL/dC or a pixel's state behind the span is not walkable. (The positions past a tile's last composited
// one are walked like the others: finding that position first, from n_contrib,
// put a load and a barrier in front of the first batch's loads.)
template <int TS, int PX, bool FINITE>
__device__ __forceinline__ bool bwd_tile_body(const Frame& f, int tile, uint32_t first, const BwdSpan& span,
                                              const uint32_t* __restrict__ vals, const float4* __restrict__ splats,
                                              const uint2* __restrict__ rect, const uint32_t* __restrict__ offsets,
                                              const float* __restrict__ t_final, const float* __restrict__ d_image,
                                              const float* __restrict__ target, const PairRecords& out,
                                              BwdSmem<TS, PX, bwd_batch<TS>()>& sm) {
    using G = TileGeom<TS, PX>;
    constexpr int BATCH = bwd_batch<TS>();
    const int tx = tile % f.TX, ty = tile / f.TX;
    const float ox = (float)(tx * TS), oy = (float)(ty * TS);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const FloatSplats sp{splats};
    const auto slot_of = [offsets](uint32_t g) { return __ldg(offsets + g); };
    // the span as batches from its front, the last one taken first
    const uint32_t begin = first + span.lo, len = span.hi - span.lo;
    if (len == 0) return true;
    uint32_t at = (len - 1) / BATCH * BATCH;
    uint32_t g0 = first_value<G, BATCH>(vals, begin + at, begin + len);
    init_null_splat(sm.rec, BATCH);
    BwdPixels<TS, PX> B;
    bool pixels_ok;
    {
        int ix, iy0;
        G::pixel(warp, lane, ix, iy0);
        float tf[PX], bf[PX], dc[PX][3];
        bool inside[PX];
        const int gx = tx * TS + ix, gy0 = ty * TS + iy0;
        // t_final before dL/dC: both are looked at below, and one wait serves
        // both (behind it, a step of short lists took 358 us, not 346)
#pragma unroll
        for (int k = 0; k < PX; ++k) {
            inside[k] = gx < f.W && gy0 + k < f.H;
            tf[k] = inside[k] ? t_final[(size_t)(gy0 + k) * f.W + gx] : 0.f;
        }
        pixels_ok = load_dc<PX>(f, gx, gy0, d_image, target, dc);
#pragma unroll
        for (int k = 0; k < PX; ++k) {
            bf[k] = dot3(f.bg, dc[k]);
            if (span.states) {
                const float2* st = span.states + (size_t)threadIdx.x * PX + k;
                for (uint32_t s = span.nseg - 1; s > span.seg; --s) {
                    const float2 v = __ldg(st + (size_t)s * (TS * TS));
                    bf[k] = fmaf(v.x, bf[k], v.y);
                }
                if (span.seg + 1 < span.nseg) {
                    float t = inside[k] ? 1.f : 0.f;
                    for (uint32_t s = 0; s <= span.seg; ++s) t *= __ldg(st + (size_t)s * (TS * TS)).x;
                    tf[k] = t;
                }
            }
            // (b stays between what lies behind and the colours projected on
            // dL/dC, so the state is looked at only once)
            pixels_ok = pixels_ok && fabsf(bf[k]) < kBehindMost && fabsf(tf[k]) < 2.f;
        }
        B.init(lane, ix, iy0, inside, tf, bf, dc, sm.dC[G::sub_block(warp, lane)]);
    }
    for (;;) {
        const int cnt = (int)min((uint32_t)BATCH, len - at);
        __syncthreads();
        const bool ok = stage_batch<G, true>(f, ox, oy, tx, ty, begin + at, cnt, g0, vals, sp, rect, slot_of, sm.rec,
                                             sm.mask, sm.slot);
        const bool more = at != 0;
        at -= more ? BATCH : 0;
        if (more) g0 = first_value<G, BATCH>(vals, begin + at, begin + at + BATCH);
        if (!__syncthreads_and(ok && pixels_ok) && FINITE) return false;
        B.template batch<FINITE>(sm, cnt, warp, lane, out);
        if (!more) return true;
    }
}

// Item i of a backward: i < split.max the i-th segment of the long lists, then
// the tiles in the order given, those with long lists left out. first: where
// the tile's list starts. Returns false for an item that does not exist.
__device__ __forceinline__ bool bwd_item(const TileOrder& o, const uint2* __restrict__ ranges, uint32_t i, int npix,
                                         uint32_t& tile, uint32_t& first, BwdSpan& span) {
    span.states = nullptr;
    span.seg = 0;
    span.nseg = 1;
    const uint32_t seg_len = o.max_split ? __ldg(o.head + 1) : ~0u;
    if (i < o.max_split) {
        if (i >= __ldg(o.head)) return false;
        const uint2 it = __ldg(o.split + i);
        tile = it.x & ((1u << kSplitTileBits) - 1u);
        const uint2 range = ranges[tile];
        const uint32_t len = range.y - range.x;
        first = range.x;
        span.seg = it.x >> kSplitTileBits;
        span.nseg = (len + seg_len - 1) / seg_len;
        span.lo = span.seg * seg_len;
        span.hi = min(span.lo + seg_len, len);
        span.states = o.states + (size_t)it.y * npix;
        return true;
    }
    tile = o.order ? __ldg(o.order + (i - o.max_split)) : i - o.max_split;
    const uint2 range = ranges[tile];
    first = range.x;
    span.lo = 0;
    span.hi = range.y - range.x;
    return span.hi <= seg_len;
}

}  // namespace ws
