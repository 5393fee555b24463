// Segmented variant of the wait-free radix sort for keys whose high bits are
// a small segment id (the tile) and whose low 31 bits are a sub-key (the
// view depth), as the renderer packs them (§3.3).
//
// The result is the same stable sort of the whole key as the plain LSD sort:
//   1. partition: the wait-free LSD passes of ws_sort.cu over the segment
//      bits [31, end_bit) only. Being stable, they leave each segment's keys
//      in input order.
//   2. bounds:    start[s] = first position whose segment id is >= s, for
//      every s in [0, 2^(end_bit - 31)], by searches of the partitioned keys.
//   3. local:     every segment is sorted by its sub-key bits [begin_bit, 31)
//      on chip, positions breaking ties, so equal sub-keys keep their input
//      order: a warp sorts one of at most 256 or 512 keys (alone_cap) with a
//      bitonic network in registers, a block one of at most 2,048 (256 threads) or
//      16,384 (1,024 threads) through buckets in shared memory or, where the
//      sub-keys crowd together, with counting passes over the list of their
//      positions, and one of more keys with chunked 8-bit passes over global
//      memory, ranked with warp ballots, skipping a pass whose digit is the
//      same for every key. The network sorts 32-bit words: the sub-key's
//      distance from the segment's smallest, cut to the leading bits that
//      fit, above the position in the segment; where bits were cut off, an
//      exchange of neighbours by the whole sub-key or two more networks put
//      right what they would have decided (warp_sort).
// A stable partition by the high bits followed by a stable sort of each
// segment by the low bits orders the pairs exactly as the full-key LSD
// sort does, ties included. There are no global atomics and no block waits
// on another: each segment belongs to one block.
//
// The local sorts are bound by instruction issue where segments fill the chip
// and by a segment's chain of dependent steps where they do not. 64-bit words
// (the whole sub-key above the position) took the network two shuffles, a
// two-part comparison and two selects an element and stage against a shuffle
// and a minimum or maximum.
#include <atomic>

#include "ws_common.cuh"
#include "ws_kernels.cuh"

namespace ws {

namespace {

constexpr int kSegThreads = 256;      // a block of a warp's segments, or of one segment of at most 2,048 keys
constexpr int kHugeThreads = 1024;     // a block of one larger segment
constexpr int kSegWarps = kSegThreads / kWarp;
constexpr int kWarpItems = 16;
constexpr int kWarpCap = kWarp * kWarpItems;      // keys a warp sorts alone
// keys that a block of THREADS sorts in shared memory, or takes at a time of a
// larger segment
template <int THREADS>
__host__ __device__ constexpr int seg_items() { return THREADS == 1024 ? 16 : 8; }
template <int THREADS>
__host__ __device__ constexpr int block_cap() { return THREADS * seg_items<THREADS>(); }
constexpr int kLocalBits = 8;
constexpr int kLocalRadix = 1 << kLocalBits;
constexpr int kSplitBit = 31;                     // segment id above, sub-key below
constexpr int kMaxSegBits = 24;

// start[s], the first position whose segment is >= s, for s in [0, nseg], and
// the same boundaries as [start, end) per tile (the local sort keeps every
// segment in place). Eight lanes search one boundary, each round splitting
// the remaining range in nine: seven rounds of dependent loads for 1M keys
// whatever their distribution, and only the probed sectors are read. A pass
// over all keys that compares neighbours read 8.9 MB and took 9.5 us on the
// 1080p / 1M frame.
constexpr int kBoundLanes = 8;

__global__ void __launch_bounds__(256)
k_seg_bounds(const uint64_t* __restrict__ keys, const uint32_t* __restrict__ num_keys, uint32_t cap,
             uint32_t seg_mask, uint32_t nseg, uint32_t* __restrict__ start, uint2* __restrict__ ranges,
             uint32_t ntiles) {
    pdl_wait();
    const uint32_t s = (blockIdx.x * 256u + threadIdx.x) / kBoundLanes;
    const uint32_t lane = threadIdx.x % kBoundLanes;
    const uint32_t gshift = threadIdx.x & 31u & ~(kBoundLanes - 1u);
    const uint32_t n = min(*num_keys, cap);
    // the answer lies in [lo, hi]; keys before lo are < s, keys from hi on >= s
    uint32_t lo = 0, hi = s == 0 ? 0u : n;
    if (s > nseg) lo = hi = 0;
    while (__any_sync(kFull, lo < hi)) {
        const uint32_t len = hi - lo;
        // probes lo + k len / 9 for k = 1 .. 8 (all below hi when lo < hi)
        const uint32_t pos = lo + (uint32_t)(((uint64_t)len * (lane + 1u)) / (kBoundLanes + 1u));
        const bool below = lo < hi && ((uint32_t)(__ldg(keys + pos) >> kSplitBit) & seg_mask) < s;
        const uint32_t c = __popc((__ballot_sync(kFull, below) >> gshift) & ((1u << kBoundLanes) - 1u));
        if (lo < hi) {
            const uint32_t nlo = c == 0 ? lo : lo + (uint32_t)(((uint64_t)len * c) / (kBoundLanes + 1u)) + 1u;
            const uint32_t nhi = c == kBoundLanes ? hi : lo + (uint32_t)(((uint64_t)len * (c + 1u)) / (kBoundLanes + 1u));
            lo = nlo;
            hi = nhi;
        }
    }
    if (lane == 0 && s <= nseg) {
        start[s] = s == nseg ? n : lo;
        const uint32_t p = s == nseg ? n : lo;
        if (ranges) {
            if (s < ntiles) ranges[s].x = p;
            if (s >= 1 && s - 1 < ntiles) ranges[s - 1].y = p;
        }
    }
}

__device__ __forceinline__ uint32_t sub_key(uint64_t k, int begin_bit, uint32_t sub_mask) {
    return (uint32_t)(k >> begin_bit) & sub_mask;
}

__device__ __forceinline__ uint32_t warp_and(uint32_t v) {
    for (int o = 16; o > 0; o >>= 1) v &= __shfl_xor_sync(kFull, v, o);
    return v;
}

__device__ __forceinline__ uint32_t warp_or(uint32_t v) {
    for (int o = 16; o > 0; o >>= 1) v |= __shfl_xor_sync(kFull, v, o);
    return v;
}

// Rank items k < kn of this warp (input order k*32 + lane) among equal
// digits: rnk = earlier equal digits of the warp; cnt[d] += the warp's count.
template <int kSegItems>
__device__ __forceinline__ void warp_rank(const uint64_t (&key)[kSegItems], int kn, int valid_base, int n,
                                          int shift, uint32_t mask, uint32_t* cnt, uint32_t (&rnk)[kSegItems]) {
    const int lane = threadIdx.x & 31;
    const uint32_t lt = lanemask_lt();
#pragma unroll
    for (int k = 0; k < kSegItems; ++k) {
        if (k >= kn) break;
        const bool ok = valid_base + k * kWarp + lane < n;
        const uint32_t d = ok ? (uint32_t)(key[k] >> shift) & mask : 0u;
        const uint32_t peers = warp_match_digit<kLocalBits>(d, ok);
        // every lane of a digit group reads the group's running count (one
        // broadcast address per group); its first lane then advances it
        const uint32_t prior = ok ? cnt[d] : 0u;
        rnk[k] = prior + __popc(peers & lt);
        __syncwarp();  // every read before the update
        if (ok && (peers & lt) == 0u) cnt[d] = prior + __popc(peers);
        __syncwarp();
    }
}

// Sort word of the element at position `idx` of its segment: its sub-key less
// the segment's smallest, without the lowest `cut` bits, above the position.
__device__ __forceinline__ uint32_t sort_word(uint32_t sub, uint32_t least, int cut, int idx_bits, uint32_t idx) {
    return (((sub - least) >> cut) << idx_bits) | idx;
}

// Bits to cut off so that `range` (largest less smallest sub-key) fits above
// idx_bits of position.
__device__ __forceinline__ int cut_bits(uint32_t range, int idx_bits) {
    return max(0, 32 - __clz(range) - (32 - idx_bits));
}

// Bitonic sorting network over the warp's 32*K distinct words, element
// e = lane*K + k in register k of lane `lane`; ascending on return. In the
// phase of runs of `size`, the lanes of descending runs hold their words
// complemented, so that every exchange is an ascending one.
template <int K>
__device__ __forceinline__ void warp_bitonic(uint32_t (&v)[K]) {
    const int lane = threadIdx.x & 31;
    const int lk = lane * K;
    constexpr int N = kWarp * K;
#pragma unroll
    for (int size = 2; size <= N; size <<= 1) {
        // complement where the run's direction differs from the last phase's
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const bool down = ((lk + k) & size) != 0;
            const bool was = size > 2 && ((lk + k) & (size >> 1)) != 0;
            v[k] ^= down != was ? ~0u : 0u;
        }
#pragma unroll
        for (int j = size >> 1; j > 0; j >>= 1) {
            if (j < K) {  // partner in the same lane
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    if (k & j) continue;
                    const uint32_t x = v[k], y = v[k | j];
                    v[k] = min(x, y);
                    v[k | j] = max(x, y);
                }
            } else {  // partner in lane ^ (j / K), same register
                const bool low = (lk & j) == 0;
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const uint32_t o = __shfl_xor_sync(kFull, v[k], j / K);
                    v[k] = low ? min(v[k], o) : max(v[k], o);
                }
            }
        }
    }
}

// Index of element e in a warp's list of sorted positions: one padding entry
// after every 16, so that lane l's entries l*K .. l*K + K - 1 and the
// consecutive entries of the way back fall in few banks.
__device__ __forceinline__ int spad(int e) { return e + (e >> 4); }

// Puts a warp's list of positions right where the cut bits would have decided:
// odd-even exchanges of neighbours by (sub-key, position). The list is sorted
// but for runs of equal sort words, most of them pairs, so a round or two will
// do; returns whether kFixRounds rounds left every neighbour in order.
constexpr int kFixRounds = 4;

template <typename Order>
__device__ __forceinline__ bool fix_order(uint16_t* list, int n, int lane, Order sub_of) {
    for (int round = 0; round < kFixRounds; ++round) {
        bool swapped = false;
        for (int odd = 0; odd < 2; ++odd) {
            for (int q = 2 * lane + odd; q + 1 < n; q += 2 * kWarp) {
                const uint16_t a = list[spad(q)], b = list[spad(q + 1)];
                const uint32_t sa = sub_of(a), sb = sub_of(b);
                if (sa > sb || (sa == sb && a > b)) {
                    list[spad(q)] = b;
                    list[spad(q + 1)] = a;
                    swapped = true;
                }
            }
            __syncwarp();  // the exchanges before the next reads
        }
        if (!__any_sync(kFull, swapped)) return true;
    }
    return false;
}

// One warp sorts n <= 32*K pairs [b, b + n) of (kin, vin) into (kout, vout): by
// the leading bits of the sub-keys and an exchange of the few neighbours that
// the rest decides; where many sub-keys share their leading bits (a wall seen
// head-on behind one near splat) the network runs twice more, over the cut
// bits and then, stably, over the leading ones.
template <int K>
__device__ __forceinline__ void warp_sort(const uint64_t* kin, const uint32_t* vin, uint64_t* kout, uint32_t* vout,
                                          uint32_t b, int n, int begin_bit, uint16_t* list) {
    const int lane = threadIdx.x & 31;
    const uint32_t sub_mask = (1u << (kSplitBit - begin_bit)) - 1u;
    constexpr int idx_bits = K == 1 ? 5 : (K == 2 ? 6 : (K == 4 ? 7 : (K == 8 ? 8 : 9)));
    constexpr uint32_t kIdxMask = (1u << idx_bits) - 1u;
    const auto sub_of = [&](uint32_t i) { return sub_key(__ldg(kin + b + i), begin_bit, sub_mask); };
    uint32_t v[K];
    uint32_t least = ~0u, most = 0u;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int idx = k * kWarp + lane;
        v[k] = idx < n ? sub_of(idx) : 0u;
        if (idx < n) {
            least = min(least, v[k]);
            most = max(most, v[k]);
        }
    }
    least = __reduce_min_sync(kFull, least);
    most = __reduce_max_sync(kFull, most);
    const int cut = cut_bits(most - least, idx_bits);
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int idx = k * kWarp + lane;
        // past the end: the largest words (the position makes them distinct)
        v[k] = idx < n ? sort_word(v[k], least, cut, idx_bits, (uint32_t)idx) : (~0u << idx_bits) | (uint32_t)idx;
    }
    // pass 0: leading bits; 1: the cut bits; 2: leading bits over pass 1's order
#pragma unroll 1
    for (int pass = 0;; ++pass) {
        warp_bitonic<K>(v);
        if (pass == 2) {  // places in pass 1's order -> positions
#pragma unroll
            for (int k = 0; k < K; ++k) v[k] = list[spad((int)(v[k] & kIdxMask))];
            __syncwarp();  // every read before the writes
        }
#pragma unroll
        for (int k = 0; k < K; ++k) list[spad(lane * K + k)] = (uint16_t)(v[k] & kIdxMask);
        __syncwarp();
        if (pass == 2 || (pass == 0 && (cut == 0 || fix_order(list, n, lane, sub_of)))) break;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int idx = k * kWarp + lane;
            v[k] = (~0u << idx_bits) | (uint32_t)idx;
            if (idx < n) {
                const uint32_t d = sub_of(pass == 0 ? (uint32_t)idx : list[spad(idx)]) - least;
                v[k] = ((pass == 0 ? d & ((1u << cut) - 1u) : d >> cut) << idx_bits) | (uint32_t)idx;
            }
        }
        __syncwarp();
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int p = k * kWarp + lane;
        if (p < n) {
            const uint32_t src = list[spad(p)];
            kout[b + p] = __ldg(kin + b + src);
            vout[b + p] = __ldg(vin + b + src);
        }
    }
}

// The block sorts n <= K THREADS pairs through 8 THREADS buckets in shared
// memory: the sub-keys' range is split over the buckets, the keys stand
// grouped by bucket after one counting pass, and each finds its place among
// its bucket's few by comparing with them. About 50 instructions a key and a
// dozen barriers, where the counting passes take up to four rounds of ballots
// and scans. Comparisons are of whole sub-keys, then positions, so the result
// is the stable order whatever order the counting's atomic additions ran in.
// The buckets are split evenly over three intervals (see bucket_of): split
// over the whole range alone, a few far splats left most keys of a clustered
// scene in few buckets. Returns false, with nothing written, when a bucket
// holds more than kBucketMost keys (sub-keys that crowd together all the
// same): the caller then sorts by the counting passes, whose work does not
// depend on the distribution. 64 of them: a 417 x 473 frame of dense tiles
// took 65.0 us for compaction and sort, 67.1 with 32, 74 with 16.
// smem: 6 K THREADS bytes of sub-keys and positions and 16 THREADS + 2 of
// buckets, at most bucket_smem of the block's largest K. The sorted pairs are
// staged there (8 K THREADS) and leave in full sectors; they are read a second
// time in input order, where gathering them in sorted order read a sector for
// each key and each value.
// Compaction and sort, us, by three passes over cut words and with blocks of
// up to 8,192 keys / by buckets and up to 16,384: 64 views / 2M 7,460 / 6,473;
// 2160p / 6M 415 / 383; 288 tiles of 2,987 keys on average 157 / 79; the sort
// of 4M pairs in 8,192 segments 192 / 175. The same buckets for a warp's
// segments lost to the network (1080p / 1M 82 against 69 us): 16 keys a lane
// in turn through shared memory is the longer chain.
constexpr uint32_t kBucketMost = 64;

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

template <int THREADS, int K>
__host__ __device__ constexpr int bucket_smem() { return 8 * K * THREADS + 16; }
static_assert(bucket_smem<1, 8>() >= 6 * 8 + 16 + 2, "sub-keys, positions and buckets of the largest K, 8 or more");

template <int THREADS, int K>
__device__ __forceinline__ bool bucket_sort(const uint64_t* kin, const uint32_t* vin, uint64_t* kout, uint32_t* vout,
                                            uint32_t b, int n, int begin_bit, unsigned char* smem, uint32_t* red) {
    constexpr int kBuckets = 8 * THREADS;
    constexpr int kOwn = kBuckets / THREADS;  // buckets a thread owns
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    uint32_t* s_word = reinterpret_cast<uint32_t*>(smem);             // sub-keys, grouped by bucket
    uint16_t* s_idx = reinterpret_cast<uint16_t*>(s_word + K * THREADS);  // and their positions
    uint16_t* s_start = s_idx + K * THREADS;  // counts, then first places; the last one is n
    uint32_t* s_pair = reinterpret_cast<uint32_t*>(s_start);
    const uint32_t sub_mask = (1u << (kSplitBit - begin_bit)) - 1u;
    uint32_t v[K], at[K];
    uint32_t least = ~0u, most = 0u;
    float total = 0.0f;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int idx = k * THREADS + t;
        v[k] = idx < n ? sub_key(__ldg(kin + b + idx), begin_bit, sub_mask) : 0u;
        if (idx < n) {
            least = min(least, v[k]);
            most = max(most, v[k]);
            total += (float)v[k];
        }
    }
#pragma unroll
    for (int k = 0; k < kOwn / 2; ++k) s_pair[k * THREADS + t] = 0u;
    least = __reduce_min_sync(kFull, least);
    most = __reduce_max_sync(kFull, most);
    total = warp_sum(total);
    if (lane == 0) {
        red[3 * warp] = least;
        red[3 * warp + 1] = most;
        red[3 * warp + 2] = __float_as_uint(total);
    }
    __syncthreads();
    total = 0.0f;
#pragma unroll
    for (int w = 0; w < THREADS / kWarp; ++w) {
        least = min(least, red[3 * w]);
        most = max(most, red[3 * w + 1]);
        total += __uint_as_float(red[3 * w + 2]);
    }
    if (least == most) {  // in order already
        for (int i = t; i < n; i += THREADS) {
            kout[b + i] = __ldg(kin + b + i);
            vout[b + i] = __ldg(vin + b + i);
        }
        return true;
    }
    const float mean = total / (float)n;
    float dev = 0.0f;
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (k * THREADS + t < n) dev += fabsf((float)v[k] - mean);
    dev = warp_sum(dev);
    constexpr int kDevs = 3 * (THREADS / kWarp);
    if (lane == 0) red[kDevs + warp] = __float_as_uint(dev);
    __syncthreads();
    dev = 0.0f;
#pragma unroll
    for (int w = 0; w < THREADS / kWarp; ++w) dev += __uint_as_float(red[kDevs + w]);
    dev = dev / (float)n + 1.0f;
    // 1/2 of the buckets for mean +- 2 dev, 1/4 for +- 5 dev, 1/4 for the whole
    // range. Every step is monotone under rounding, so the order of sub-keys is
    // kept, which is all the buckets need.
    const float a1 = 0.25f / dev, a2 = 0.1f / dev, a3 = 1.0f / ((float)(most - least) + 1.0f);
    const float o1 = 0.5f - mean * a1, o2 = 0.5f - mean * a2, o3 = -(float)least * a3;
    auto bucket_of = [&](uint32_t x) {
        const float f = (float)x;
        float u = 0.25f * __saturatef(fmaf(f, a3, o3));
        u = fmaf(0.25f, __saturatef(fmaf(f, a2, o2)), u);
        u = fmaf(0.5f, __saturatef(fmaf(f, a1, o1)), u);
        return min((uint32_t)kBuckets - 1u, (uint32_t)(u * (float)kBuckets));
    };
#pragma unroll
    for (int k = 0; k < K; ++k) {
        at[k] = 0u;
        if (k * THREADS + t < n) {
            const uint32_t bk = bucket_of(v[k]);
            const uint32_t half = (bk & 1u) * 16u;
            at[k] = bk | ((atomicAdd(s_pair + (bk >> 1), 1u << half) >> half) << 16);
        }
    }
    __syncthreads();
    // counts -> first places: thread t owns kOwn in a row
    uint32_t c[kOwn / 2];
    uint32_t sum = 0u, crowd = 0u;
#pragma unroll
    for (int k = 0; k < kOwn / 2; ++k) {
        c[k] = s_pair[t * (kOwn / 2) + k];
        sum += (c[k] & 0xffffu) + (c[k] >> 16);
        crowd = max(crowd, max(c[k] & 0xffffu, c[k] >> 16));
    }
    if (__syncthreads_or(crowd > kBucketMost)) return false;
    uint32_t all;
    uint32_t first = block_exclusive_scan<THREADS>(sum, red, &all);
#pragma unroll
    for (int k = 0; k < kOwn / 2; ++k) {
        const uint32_t second = first + (c[k] & 0xffffu);
        s_pair[t * (kOwn / 2) + k] = first | (second << 16);
        first = second + (c[k] >> 16);
    }
    if (t == 0) s_start[kBuckets] = (uint16_t)n;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int idx = k * THREADS + t;
        if (idx < n) {
            const uint32_t p = s_start[at[k] & 0xffffu] + (at[k] >> 16);
            s_word[p] = v[k];
            s_idx[p] = (uint16_t)idx;
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int idx = k * THREADS + t;
        if (idx < n) {
            const uint32_t bk = at[k] & 0xffffu;
            const uint32_t p0 = s_start[bk], p1 = s_start[bk + 1], own = p0 + (at[k] >> 16);
            uint32_t rank = p0;
            for (uint32_t p = p0; p < p1; ++p) {
                const uint32_t w = s_word[p];
                if (w < v[k]) ++rank;
                if (w == v[k] && p != own && s_idx[p] < (uint16_t)idx) ++rank;
            }
            at[k] = rank;
        }
    }
    __syncthreads();
    uint64_t* s_key = reinterpret_cast<uint64_t*>(smem);
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int idx = k * THREADS + t;
        if (idx < n) s_key[at[k]] = __ldg(kin + b + idx);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int idx = k * THREADS + t;
        if (idx < n) kout[b + idx] = s_key[idx];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int idx = k * THREADS + t;
        if (idx < n) s_word[at[k]] = __ldg(vin + b + idx);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int idx = k * THREADS + t;
        if (idx < n) vout[b + idx] = s_word[idx];
    }
    return true;
}

// Block-wide AND / OR of one value per thread.
template <int THREADS>
__device__ __forceinline__ uint32_t block_varying(uint32_t a, uint32_t o, uint32_t* red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    a = warp_and(a);
    o = warp_or(o);
    __syncthreads();
    if (lane == 0) {
        red[2 * warp] = a;
        red[2 * warp + 1] = o;
    }
    __syncthreads();
    uint32_t ra = ~0u, ro = 0u;
#pragma unroll
    for (int w = 0; w < THREADS / kWarp; ++w) {
        ra &= red[2 * w];
        ro |= red[2 * w + 1];
    }
    return ra ^ ro;
}

// The block sorts n <= block_cap pairs by stable 8-bit LSD passes over the list
// of their positions, at most four, skipping those whose digit is the same
// for every key; with kn = ceil(n / THREADS), element w*32*kn + k*32 + lane of the
// list lives in lane `lane` of warp w, item k. s_sub: the sub-keys by position;
// s_cnt: THREADS / 32 rows of 256 counters.
constexpr int kCtaDigit = 8;
constexpr int kCtaRadix = 1 << kCtaDigit;

template <int THREADS>
__device__ __forceinline__ void block_sort_smem(const uint64_t* kin, const uint32_t* vin, uint64_t* kout,
                                                uint32_t* vout, uint32_t b, int n, int begin_bit, uint32_t* s_sub,
                                                uint16_t* s_list, uint16_t* s_cnt, uint32_t* red) {
    constexpr int kSegItems = seg_items<THREADS>();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // every warp takes kn consecutive runs of 32 (input order = warp, item, lane)
    const int kn = (n + THREADS - 1) / THREADS;
    const int wbase = warp * kWarp * kn;
    const uint32_t sub_mask = (1u << (kSplitBit - begin_bit)) - 1u;
    uint32_t all_and = ~0u, all_or = 0u;
    for (int i = threadIdx.x; i < n; i += THREADS) {
        const uint32_t x = sub_key(__ldg(kin + b + i), begin_bit, sub_mask);
        s_sub[i] = x;
        all_and &= x;
        all_or |= x;
    }
    const uint32_t varying = block_varying<THREADS>(all_and, all_or, red);  // (its barriers publish s_sub)
    uint32_t at[kSegItems];  // position, and the digit's count and rank in the pass
#pragma unroll
    for (int k = 0; k < kSegItems; ++k) at[k] = (uint32_t)(wbase + k * kWarp + lane);
    const uint32_t lt = lanemask_lt();
    uint16_t* cnt = s_cnt + warp * kCtaRadix;
    for (int shift = 0; shift < kSplitBit - begin_bit; shift += kCtaDigit) {
        if (((varying >> shift) & (kCtaRadix - 1)) == 0u) continue;
        __syncthreads();  // the last pass's reads of the list and counters
        reinterpret_cast<uint4*>(cnt)[lane] = make_uint4(0u, 0u, 0u, 0u);
        __syncwarp();
        uint16_t rnk[kSegItems];
#pragma unroll
        for (int k = 0; k < kSegItems; ++k) {
            if (k >= kn) break;
            const bool ok = wbase + k * kWarp + lane < n;
            const uint32_t dg = ok ? (s_sub[at[k]] >> shift) & (kCtaRadix - 1) : 0u;
            const uint32_t peers = warp_match_digit<kCtaDigit>(dg, ok);
            const uint32_t prior = cnt[dg];
            rnk[k] = (uint16_t)(prior + __popc(peers & lt));
            __syncwarp();
            if (ok && (peers & lt) == 0u) cnt[dg] = (uint16_t)(prior + __popc(peers));
            __syncwarp();
        }
        __syncthreads();
        // counts -> first positions, by digit and then warp: thread t owns
        // digit t of the first 256 threads
        uint32_t run = 0;
        if (threadIdx.x < kCtaRadix)
            for (int w = 0; w < THREADS / kWarp; ++w) run += s_cnt[w * kCtaRadix + threadIdx.x];
        uint32_t all;
        uint32_t first = block_exclusive_scan<THREADS>(run, red, &all);
        if (threadIdx.x < kCtaRadix) {
            for (int w = 0; w < THREADS / kWarp; ++w) {
                const uint32_t c = s_cnt[w * kCtaRadix + threadIdx.x];
                s_cnt[w * kCtaRadix + threadIdx.x] = (uint16_t)first;
                first += c;
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kSegItems; ++k) {
            if (k >= kn) break;
            if (wbase + k * kWarp + lane < n)
                s_list[cnt[(s_sub[at[k]] >> shift) & (kCtaRadix - 1)] + rnk[k]] = (uint16_t)at[k];
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kSegItems; ++k) {
            if (k >= kn) break;
            const int idx = wbase + k * kWarp + lane;
            if (idx < n) at[k] = s_list[idx];
        }
    }
#pragma unroll
    for (int k = 0; k < kSegItems; ++k) {
        if (k >= kn) break;
        const int idx = wbase + k * kWarp + lane;
        if (idx < n) {
            kout[b + idx] = __ldg(kin + b + at[k]);
            vout[b + idx] = __ldg(vin + b + at[k]);
        }
    }
}

// The block sorts any number of pairs through global memory, 8 THREADS at a
// time: per pass a histogram sweep, then chunks in order, each scattered to its
// digit's running offset. One block works alone, bound by its chain of loads,
// ballots and barriers: the histogram therefore takes one addition a key, no
// ranks, which also leaves the 256-thread block's 64 registers without spills
// (4M pairs, a fifth of them in 20 segments of 40,000: 855-867 us, in one run of
// four 698, with the ranks, 694-701 without; a half in 200 segments of 10,000:
// 357-368 -> 300-335). Ping-pongs between the two buffers' [b, b + n);
// the result ends in (kout, vout). Loads here are plain (not read-only
// cache): the block reads what it wrote, ordered by __syncthreads.
template <int THREADS>
__device__ void block_sort_global(uint64_t* kin, uint32_t* vin, uint64_t* kout, uint32_t* vout, uint32_t b,
                                  uint32_t n, int begin_bit, uint32_t (*cnt)[kLocalRadix], uint32_t* off,
                                  uint32_t* red) {
    constexpr int kSegItems = 8;
    constexpr uint32_t kStep = THREADS * kSegItems;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int wbase = warp * kWarp * kSegItems;
    const uint32_t sub_mask = (1u << (kSplitBit - begin_bit)) - 1u;
    uint32_t all_and = ~0u, all_or = 0u;
    for (uint32_t c0 = 0; c0 < n; c0 += kStep) {
#pragma unroll
        for (int k = 0; k < kSegItems; ++k) {
            const uint32_t idx = c0 + wbase + k * kWarp + lane;
            if (idx < n) {
                const uint32_t s = sub_key(kin[b + idx], begin_bit, sub_mask);
                all_and &= s;
                all_or |= s;
            }
        }
    }
    const uint32_t varying = block_varying<THREADS>(all_and, all_or, red);
    uint64_t* sk = kin + b;
    uint32_t* sv = vin + b;
    uint64_t* dk = kout + b;
    uint32_t* dv = vout + b;
    bool in_out = false;  // data currently in (kout, vout)?
    for (int shift = begin_bit; shift < kSplitBit; shift += kLocalBits) {
        const int bits = kSplitBit - shift < kLocalBits ? kSplitBit - shift : kLocalBits;
        const uint32_t mask = (1u << bits) - 1u;
        if (((varying >> (shift - begin_bit)) & mask) == 0u) continue;
        // digit totals of the segment -> running offsets (integer additions:
        // the counts do not depend on their order)
        if (threadIdx.x < kLocalRadix) off[threadIdx.x] = 0u;
        __syncthreads();
#pragma unroll 8
        for (uint32_t i = threadIdx.x; i < n; i += THREADS) atomicAdd(&off[(uint32_t)(sk[i] >> shift) & mask], 1u);
        __syncthreads();
        {
            const int d = threadIdx.x;  // the first 256 threads are the digits
            uint32_t all;
            const uint32_t t = block_exclusive_scan<THREADS>(d < kLocalRadix ? off[d] : 0u, red, &all);
            if (d < kLocalRadix) off[d] = t;
        }
        __syncthreads();
        for (uint32_t c0 = 0; c0 < n; c0 += kStep) {
            const int rem = (int)min(n - c0, kStep);
            const int kn = rem > wbase ? ((rem - wbase + kWarp - 1) / kWarp < kSegItems
                                              ? (rem - wbase + kWarp - 1) / kWarp
                                              : kSegItems)
                                       : 0;
            for (int i = threadIdx.x; i < (THREADS / kWarp) * kLocalRadix; i += THREADS) (&cnt[0][0])[i] = 0u;
            __syncthreads();
            uint64_t key[kSegItems];
            uint32_t val[kSegItems];
#pragma unroll
            for (int k = 0; k < kSegItems; ++k) {
                const int idx = wbase + k * kWarp + lane;
                const bool ok = k < kn && idx < rem;
                key[k] = ok ? sk[c0 + idx] : 0ull;
                val[k] = ok ? sv[c0 + idx] : 0u;
            }
            uint32_t rnk[kSegItems];
            warp_rank(key, kn, wbase, rem, shift, mask, cnt[warp], rnk);
            __syncthreads();
            // per-warp prefix within the chunk (no digit starts: the
            // running offsets place the chunk)
            const int d = threadIdx.x;
            uint32_t run = 0;
            if (d < kLocalRadix) {
#pragma unroll
                for (int w = 0; w < (THREADS / kWarp); ++w) {
                    const uint32_t c = cnt[w][d];
                    cnt[w][d] = run;
                    run += c;
                }
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < kSegItems; ++k) {
                if (k >= kn) break;
                if (wbase + k * kWarp + lane < rem) {
                    const uint32_t dg = (uint32_t)(key[k] >> shift) & mask;
                    const uint32_t pos = off[dg] + cnt[warp][dg] + rnk[k];
                    dk[pos] = key[k];
                    dv[pos] = val[k];
                }
            }
            __syncthreads();
            if (d < kLocalRadix) off[d] += run;
        }
        __syncthreads();
        uint64_t* tk = sk; sk = dk; dk = tk;
        uint32_t* tv = sv; sv = dv; dv = tv;
        in_out = !in_out;
    }
    if (!in_out) {  // an even number of passes ran: copy into (kout, vout)
        for (uint32_t i = threadIdx.x; i < n; i += THREADS) {
            kout[b + i] = kin[b + i];
            vout[b + i] = vin[b + i];
        }
    }
}

// Shared memory of a block that sorts one segment: the sub-keys, positions and
// counters of the passes over positions, the counters of the passes over
// global memory, or the buckets.
template <int THREADS>
struct SegSmem {
    static constexpr int kWordBytes = block_cap<THREADS>() * 4;
    static constexpr int kListBytes = block_cap<THREADS>() * 2;
    static constexpr int kBytes = kWordBytes + kListBytes + (THREADS / kWarp) * kCtaRadix * 2;
    static constexpr int kGlobalBytes = (THREADS / kWarp) * kLocalRadix * 4;
    static constexpr int kPassBytes = kBytes > kGlobalBytes ? kBytes : kGlobalBytes;
    static constexpr int kBucketBytes = bucket_smem<THREADS, seg_items<THREADS>()>();
    static constexpr int kRaw = kPassBytes > kBucketBytes ? kPassBytes : kBucketBytes;
};

// The block sorts one segment [b, b + n).
template <int THREADS>
__device__ __forceinline__ void block_sort(uint64_t* kin, uint32_t* vin, uint64_t* kout, uint32_t* vout, uint32_t b,
                                           uint32_t n, int begin_bit, unsigned char* raw, uint32_t* off,
                                           uint32_t* red) {
    if (n <= (uint32_t)block_cap<THREADS>()) {
        bool done;
        if (n <= 4 * THREADS)
            done = bucket_sort<THREADS, 4>(kin, vin, kout, vout, b, (int)n, begin_bit, raw, red);
        else if (seg_items<THREADS>() == 8 || n <= 8 * THREADS)
            done = bucket_sort<THREADS, 8>(kin, vin, kout, vout, b, (int)n, begin_bit, raw, red);
        else
            done = bucket_sort<THREADS, seg_items<THREADS>()>(kin, vin, kout, vout, b, (int)n, begin_bit, raw, red);
        if (done) return;
        __syncthreads();  // every thread is done with the shared memory
        using M = SegSmem<THREADS>;
        block_sort_smem<THREADS>(kin, vin, kout, vout, b, (int)n, begin_bit, reinterpret_cast<uint32_t*>(raw),
                                 reinterpret_cast<uint16_t*>(raw + M::kWordBytes),
                                 reinterpret_cast<uint16_t*>(raw + M::kWordBytes + M::kListBytes), red);
    } else {
        block_sort_global<THREADS>(kin, vin, kout, vout, b, n, begin_bit,
                                   reinterpret_cast<uint32_t (*)[kLocalRadix]>(raw), off, red);
    }
}

// Segment s as [b, e), clamped into [0, n].
__device__ __forceinline__ void seg_bounds(const uint32_t* __restrict__ start, uint32_t s, uint32_t n, uint32_t& b,
                                           uint32_t& e) {
    e = min(__ldg(start + s + 1), n);
    b = min(__ldg(start + s), e);
}

// The segments i, i + nblocks, i + 2 nblocks, ... (32 at most) of block i, of
// more than `above` and at most `most` keys, one after another.
template <int THREADS>
__device__ __forceinline__ void sort_own_segments(uint64_t* kin, uint32_t* vin, uint64_t* kout, uint32_t* vout,
                                                  const uint32_t* __restrict__ start, uint32_t n_all, uint32_t nseg,
                                                  uint32_t nblocks, uint32_t above, uint32_t most, int begin_bit,
                                                  unsigned char* raw, uint32_t* off, uint32_t* red) {
    uint32_t b0 = 0, e0 = 0;  // bounds of the lane's segment (every warp alike)
    const uint32_t s0 = blockIdx.x + (threadIdx.x & 31u) * nblocks;
    if (s0 < nseg) seg_bounds(start, s0, n_all, b0, e0);
    uint32_t todo = __ballot_sync(kFull, e0 - b0 > above && e0 - b0 <= most);
    while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1;
        const uint32_t b = __shfl_sync(kFull, b0, src), n = __shfl_sync(kFull, e0, src) - b;
        block_sort<THREADS>(kin, vin, kout, vout, b, n, begin_bit, raw, off, red);
        __syncthreads();  // shared memory is free for the next segment
    }
}

// Keys a warp sorts alone: 512 where there are segments enough to fill the chip
// several times over (the network's instructions a key bound the sort then),
// else 256 (a warp's chain of 45 exchanges of 16 words then leaves the chip
// waiting for the last warps, where a block of buckets is done in a third of
// the time). Compaction and sort, 512 against 256: 2160p / 6M (32,768
// segments of 263 keys on average) 383 against 399 us, 64 views / 2M (262,144 of
// 460) 6.66 against 6.70 ms; 1080p / 1M (8,192 of 140) 67.4 against 65.3, 720p /
// 500k (4,096 of 121) 47.5 against 43.2, 6 views / 300k (32,768 of 59) 153.5
// against 147.8.
__device__ __forceinline__ uint32_t alone_cap(uint32_t n, uint32_t nseg) {
    return nseg > 8192u && n >= 192u * nseg ? 512u : 256u;
}

// Blocks [0, nbig) sort the segments of more than alone_cap and at most `most` keys:
// block i those among i, i + nbig, i + 2 nbig, ..., found by one look at their
// bounds. Blocks nbig + g, g >= 0, give warp w the segment 8g + w when it
// holds 1 to alone_cap keys. The large segments come first in launch order so their
// longer sorts start early.
// nbig (big_blocks): every segment its own block up to 2,048 of them, then
// 2,048 blocks and more segments each: a block that finds nothing to do still
// costs its launch (8,192 of them 13 us of the 1080p / 1M frame's 34 us local
// sort), while a block with many large segments sorts them one after another
// (with 256 blocks for 8,192 segments of 514 keys on average, 311 us instead
// of 209 for the whole sort).
uint32_t big_blocks(uint32_t nseg) {
    const uint32_t per = nseg <= 2048u ? 1u : (nseg / 2048u < 32u ? nseg / 2048u : 32u);
    return (nseg + per - 1) / per;
}

__global__ void __launch_bounds__(kSegThreads, 4)
k_seg_sort(uint64_t* kin, uint32_t* vin, uint64_t* kout, uint32_t* vout, const uint32_t* __restrict__ start,
           const uint32_t* __restrict__ num_keys, uint32_t cap, uint32_t nseg, uint32_t nbig, uint32_t most,
           int begin_bit) {
    // One buffer, carved two ways: a block's segment, or each warp's list.
    constexpr int kListLen = kWarpCap + kWarpCap / 16;
    constexpr int kListBytes = kSegWarps * kListLen * 2;
    constexpr int kRaw = SegSmem<kSegThreads>::kRaw > kListBytes ? SegSmem<kSegThreads>::kRaw : kListBytes;
    __shared__ __align__(16) unsigned char s_raw[kRaw];
    __shared__ uint32_t s_off[kLocalRadix];
    __shared__ uint32_t s_red[4 * kSegWarps];
    const int warp = threadIdx.x >> 5;
    pdl_wait();
    const uint32_t n_all = min(*num_keys, cap);
    const uint32_t alone = alone_cap(n_all, nseg);
    if (blockIdx.x < nbig) {
        sort_own_segments<kSegThreads>(kin, vin, kout, vout, start, n_all, nseg, nbig, alone, most,
                                       begin_bit, s_raw, s_off, s_red);
        return;
    }
    const uint32_t s = (blockIdx.x - nbig) * kSegWarps + warp;
    if (s >= nseg) return;
    uint32_t b, e;
    seg_bounds(start, s, n_all, b, e);
    const int n = (int)(e - b);
    if (n == 0 || n > (int)alone) return;
    uint16_t* list = reinterpret_cast<uint16_t*>(s_raw) + warp * kListLen;
    if (n <= 32)
        warp_sort<1>(kin, vin, kout, vout, b, n, begin_bit, list);
    else if (n <= 64)
        warp_sort<2>(kin, vin, kout, vout, b, n, begin_bit, list);
    else if (n <= 128)
        warp_sort<4>(kin, vin, kout, vout, b, n, begin_bit, list);
    else if (n <= 256)
        warp_sort<8>(kin, vin, kout, vout, b, n, begin_bit, list);
    else
        warp_sort<16>(kin, vin, kout, vout, b, n, begin_bit, list);
}

// The segments of more than 2,048 keys, 1,024 threads each (up to 16,384 keys
// in shared memory). Launched where the capacity allows such segments to be
// common, kHugeMean keys or more a segment: the launch costs 3 us, and the
// 256-thread blocks of k_seg_sort, which take them otherwise, 8 passes over
// global memory.
constexpr uint32_t kHugeMean = 600;
__global__ void __launch_bounds__(kHugeThreads, 1)
k_seg_sort_huge(uint64_t* kin, uint32_t* vin, uint64_t* kout, uint32_t* vout, const uint32_t* __restrict__ start,
                const uint32_t* __restrict__ num_keys, uint32_t cap, uint32_t nseg, int begin_bit) {
    extern __shared__ __align__(16) unsigned char s_raw[];  // SegSmem<kHugeThreads>::kRaw
    __shared__ uint32_t s_off[kLocalRadix];
    __shared__ uint32_t s_red[4 * kHugeThreads / kWarp];
    pdl_wait();
    const uint32_t n_all = min(*num_keys, cap);
    sort_own_segments<kHugeThreads>(kin, vin, kout, vout, start, n_all, nseg, gridDim.x,
                                    (uint32_t)block_cap<kSegThreads>(), ~0u, begin_bit, s_raw, s_off, s_red);
}

// Scratch: [partition histograms, sized for 11-bit digits | segment starts].
size_t seg_start_offset_words(int64_t key_capacity) { return sort_scratch_bytes(key_capacity, 11) / 4; }

size_t seg_starts_words(int64_t key_capacity) {
    const size_t w = sort_scratch_bytes(key_capacity, 11) / 4;
    const size_t most = (size_t(1) << kMaxSegBits) + 1;
    return w < most ? w : most;
}

}  // namespace

size_t sort_segmented_scratch_bytes(int64_t key_capacity) {
    return (seg_start_offset_words(key_capacity) + seg_starts_words(key_capacity)) * sizeof(uint32_t);
}

bool sort_segmented_supported(int64_t key_capacity, int begin_bit, int end_bit) {
    if (begin_bit < 0 || begin_bit >= kSplitBit || end_bit <= kSplitBit || end_bit - kSplitBit > kMaxSegBits)
        return false;
    const uint64_t nseg = uint64_t(1) << (end_bit - kSplitBit);
    return nseg + 1 <= seg_starts_words(key_capacity);
}

int sort_segmented_first_digit(int end_bit, int digit_bits) {
    // Partition by the segment bits: as few passes as digits of at most
    // digit_bits bits allow, their width split evenly (13 segment bits at
    // digit_bits 8 or 9: 7 + 6); 4 bits at least.
    const int seg_bits = end_bit - kSplitBit;
    const int max_digit = digit_bits < 4 ? 4 : (digit_bits > 11 ? 11 : digit_bits);
    const int passes = (seg_bits + max_digit - 1) / max_digit;
    const int digit = (seg_bits + passes - 1) / passes;
    return digit < 4 ? 4 : digit;
}

cudaError_t launch_sort_segmented(const uint32_t* num_keys, int64_t key_capacity, int begin_bit, int end_bit,
                                  int digit_bits, uint64_t* keys, uint32_t* vals, uint64_t* keys_alt,
                                  uint32_t* vals_alt, void* scratch, int* in_alt, cudaStream_t stream,
                                  uint32_t* ranges, uint32_t ntiles, bool first_pass_done) {
    const int seg_bits = end_bit - kSplitBit;
    const int digit = sort_segmented_first_digit(end_bit, digit_bits);
    // With first_pass_done the keys already stand stably partitioned by the
    // first digit (the fused compaction): the passes start at the second.
    const int part_begin = first_pass_done ? kSplitBit + digit : kSplitBit;
    int part_alt = 0;
    cudaError_t e = cudaSuccess;
    if (part_begin < end_bit) {
        e = launch_sort(num_keys, key_capacity, part_begin, end_bit, digit, keys, vals, keys_alt, vals_alt, scratch,
                        &part_alt, stream);
        if (e != cudaSuccess) return e;
    }
    uint64_t* pk = part_alt ? keys_alt : keys;
    uint32_t* pv = part_alt ? vals_alt : vals;
    uint64_t* ok = part_alt ? keys : keys_alt;
    uint32_t* ov = part_alt ? vals : vals_alt;
    uint32_t* start = static_cast<uint32_t*>(scratch) + seg_start_offset_words(key_capacity);
    const uint32_t nseg = 1u << seg_bits;
    const uint32_t bound_blocks = (uint32_t)(((uint64_t)(nseg + 1u) * kBoundLanes + 255u) / 256u);
    e = launch_pdl(k_seg_bounds, dim3(bound_blocks), dim3(256), 0, stream, (const uint64_t*)pk, num_keys,
                   (uint32_t)key_capacity, nseg - 1u, nseg, start, reinterpret_cast<uint2*>(ranges), ntiles);
    if (e != cudaSuccess) return e;
    const bool huge = (uint64_t)key_capacity >= (uint64_t)kHugeMean * nseg &&
                      key_capacity > (int64_t)block_cap<kSegThreads>();
    if (huge) {
        constexpr int smem = SegSmem<kHugeThreads>::kRaw;
        // above the default limit: set once per device
        static std::atomic<uint64_t> configured{0};
        int dev = 0;
        e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        const uint64_t bit = uint64_t(1) << (dev & 63);
        if (!(configured.load(std::memory_order_acquire) & bit)) {
            e = cudaFuncSetAttribute(k_seg_sort_huge, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            if (e != cudaSuccess) return e;
            configured.fetch_or(bit, std::memory_order_acq_rel);
        }
        e = launch_pdl(k_seg_sort_huge, dim3(nseg <= 512u ? nseg : (nseg / 32u < 512u ? 512u : (nseg + 31u) / 32u)),
                       dim3(kHugeThreads), (size_t)smem, stream, pk, pv, ok, ov, (const uint32_t*)start, num_keys,
                       (uint32_t)key_capacity, nseg, begin_bit);
        if (e != cudaSuccess) return e;
    }
    const uint32_t nbig = big_blocks(nseg);
    e = launch_pdl(k_seg_sort, dim3(nbig + (nseg + kSegWarps - 1) / kSegWarps), dim3(kSegThreads), 0, stream, pk, pv,
                   ok, ov, (const uint32_t*)start, num_keys, (uint32_t)key_capacity, nseg, nbig,
                   huge ? (uint32_t)block_cap<kSegThreads>() : ~0u, begin_bit);
    if (e != cudaSuccess) return e;
    *in_alt = !part_alt;
    return cudaGetLastError();
}

}  // namespace ws
