// radix.cuh -- stable LSD radix sort of 32- or 64-bit keys with 32-bit values
// (digit histograms per tile, an exclusive scan of them, a stable scatter).
// Used by the banding step (band keys) and the prefix-filter candidate
// generator (index entries and candidate pairs).
#pragma once

#include "common.cuh"
#include "scan.cuh"

namespace blsh_radix {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kSortThreads = 256;
constexpr int kSortPerThread = 16;
constexpr int kSortTile = kSortThreads * kSortPerThread;   // 4096 items per CTA
constexpr int kWarps = kSortThreads / 32;

// The items are `segs` segments of seg_len each, every segment sorted by
// itself (the banding step's bands lie one after the other, so the band index
// needs no digits); a tile lies in one segment, and the histograms are laid
// out [segment][digit][tile], so that one scan gives every run its place.
struct Shape {
    long long seg_len;
    unsigned segs, tps;   // tiles per segment
};
inline Shape shape(long long seg_len, long long segs) {
    return {seg_len, (unsigned)segs, (unsigned)((seg_len + kSortTile - 1) / kSortTile)};
}

// The tile's first item, its length, and the histogram entry of its digit 0.
struct Tile {
    long long first;
    int len;
    size_t hist0;
    long long in_seg;   // first item's position in its segment
};
template <int RB>
__device__ __forceinline__ Tile tile_of(const Shape &S) {
    const unsigned seg = S.segs == 1 ? 0u : blockIdx.x / S.tps, t = blockIdx.x - seg * S.tps;
    Tile T;
    T.in_seg = (long long)t * kSortTile;
    T.first = (long long)seg * S.seg_len + T.in_seg;
    const long long left = S.seg_len - T.in_seg;
    T.len = (int)(left < kSortTile ? left : kSortTile);
    T.hist0 = ((size_t)seg << RB) * S.tps + t;
    return T;
}

// ---- stable LSD radix sort, one RB-bit digit per pass ---------------------

template <typename K, int RB>
__global__ void __launch_bounds__(kSortThreads) digit_hist_kernel(const K *__restrict__ keys, Shape S, int shift,
                                                                  uint32_t mask, uint32_t *__restrict__ hist) {
    __shared__ uint32_t h[1 << RB];
    for (int d = threadIdx.x; d < (1 << RB); d += kSortThreads) h[d] = 0;
    __syncthreads();
    const Tile T = tile_of<RB>(S);
    K k[kSortPerThread];   // all loads in flight before the first count
#pragma unroll
    for (int i = 0; i < kSortPerThread; ++i) {
        const int p = i * kSortThreads + threadIdx.x;
        k[i] = p < T.len ? __ldg(keys + T.first + p) : K(0);
    }
#pragma unroll
    for (int i = 0; i < kSortPerThread; ++i)
        if (i * kSortThreads + (int)threadIdx.x < T.len) atomicAdd(&h[(uint32_t)(k[i] >> shift) & mask], 1u);
    __syncthreads();
    for (int d = threadIdx.x; d < (1 << RB); d += kSortThreads) hist[T.hist0 + (size_t)d * S.tps] = h[d];
}

// Ranks of one warp's items among those of the same digit: 32 at a time, lanes
// holding the same digit (of RB bits) found by a ballot per bit, all rounds'
// first (they do not depend on each other), then the running counts in
// cnt[digit] (the warp's own, in shared memory).  Items past `len` (a digit
// outside the table) take no part.  __match_any_sync in the place of the
// ballots, inside the counts' chain, bound the scatter: 6.4e7 items of 8-bit
// digits 465 us a pass, 426 ahead of the chain, ballots in it 349, ahead 312.
template <int RB, int ROUNDS, typename DigitOf>
__device__ __forceinline__ void warp_ranks(uint32_t *cnt, uint32_t (&rank)[ROUNDS], DigitOf digit_of) {
    const unsigned lt = (1u << (threadIdx.x & 31)) - 1u;
    unsigned peers[ROUNDS];
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        bool ok;
        const uint32_t d = digit_of(r, ok);
        unsigned p = __ballot_sync(kFull, ok);
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            const bool set = (d >> i) & 1u;
            const unsigned with = __ballot_sync(kFull, set);
            p &= set ? with : ~with;
        }
        peers[r] = p;
    }
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        bool ok;
        const uint32_t d = digit_of(r, ok);
        const uint32_t before = ok ? cnt[d] : 0u;
        rank[r] = before + __popc(peers[r] & lt);
        __syncwarp();
        if (ok && (peers[r] & lt) == 0) cnt[d] = before + __popc(peers[r]);
        __syncwarp();
    }
}

// Scatter with stable ranks, through shared memory.  Warp w ranks the
// contiguous items [w*512, (w+1)*512) of the tile (keys loaded into registers
// up front, so that no load waits behind a ranking round); the warps' counts
// are then offset by those of lower warps, the tile's digit totals scanned,
// and every item placed in shared memory in digit order; finally consecutive
// threads write consecutive positions, so each digit's run of the tile goes
// out in coalesced stores.  Equal digits keep the tile's order (warp, then
// round, then lane), so the sort is stable.  vals_in == NULL: an item's value
// is its position in its segment.
// 6.4e7 items: 2.94 ms for three 8-bit digits of 64-bit keys (hist, scan,
// scatter) before the keys went to 32 bits, the band index out of the sort and
// the loads to the front; 0.84 ms for two digits now.  Three CTAs an SM for
// 64-bit keys too, although that costs them 116 bytes of spills: 5e7 keys, eight
// digits, 2.83 ms against 3.06 without the bound.
template <typename K, int RB>
constexpr size_t scatter_smem() {
    return (size_t)kSortTile * (sizeof(K) + sizeof(uint32_t)) + (size_t)kWarps * (1 << RB) * sizeof(uint32_t) +
           2 * (size_t)(1 << RB) * sizeof(uint32_t);
}
template <typename K, int RB>
__global__ void __launch_bounds__(kSortThreads, 3) digit_scatter_kernel(const K *__restrict__ keys_in,
                                                                     const uint32_t *__restrict__ vals_in, Shape S,
                                                                     int shift, uint32_t mask,
                                                                     const uint32_t *__restrict__ offsets,
                                                                     K *__restrict__ keys_out,
                                                                     uint32_t *__restrict__ vals_out) {
    constexpr int ND = 1 << RB;
    extern __shared__ __align__(16) unsigned char sm[];
    K *s_key = reinterpret_cast<K *>(sm);
    uint32_t *s_val = reinterpret_cast<uint32_t *>(s_key + kSortTile);
    uint32_t(*cnt)[ND] = reinterpret_cast<uint32_t(*)[ND]>(s_val + kSortTile);
    uint32_t *s_start = reinterpret_cast<uint32_t *>(cnt + kWarps);   // first position of a digit in the tile
    uint32_t *s_out = s_start + ND;                                    // its place in the output, less that
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const Tile T = tile_of<RB>(S);
    const int base = w * (kSortTile / kWarps) + lane;
    K key[kSortPerThread];
#pragma unroll
    for (int r = 0; r < kSortPerThread; ++r)
        key[r] = base + r * 32 < T.len ? __ldg(keys_in + T.first + base + r * 32) : K(0);
    for (int d = lane; d < ND; d += 32) cnt[w][d] = 0;
    __syncwarp();
    uint32_t rank[kSortPerThread];
    warp_ranks<RB, kSortPerThread>(cnt[w], rank, [&](int r, bool &ok) {
        ok = base + r * 32 < T.len;
        return (uint32_t)(key[r] >> shift) & mask;
    });
    // the items' values, in flight over the prefix sums
    uint32_t val[kSortPerThread];
#pragma unroll
    for (int r = 0; r < kSortPerThread; ++r) {
        const int p = base + r * 32;
        val[r] = !vals_in ? (uint32_t)(T.in_seg + p) : p < T.len ? __ldg(vals_in + T.first + p) : 0u;
    }
    __syncthreads();
    // per digit: exclusive prefix over warps, then the tile's digit totals
    // scanned (thread t: digits t ND/256 ..)
    constexpr int DPT = ND / kSortThreads;
    uint32_t total[DPT], sum = 0;
#pragma unroll
    for (int i = 0; i < DPT; ++i) {
        const int d = threadIdx.x * DPT + i;
        total[i] = 0;
        for (int ww = 0; ww < kWarps; ++ww) {
            const uint32_t c = cnt[ww][d];
            cnt[ww][d] = total[i];
            total[i] += c;
        }
        sum += total[i];
    }
    uint32_t start = blsh_scan::block_exclusive<uint32_t>(sum, nullptr);
#pragma unroll
    for (int i = 0; i < DPT; ++i) {
        const int d = threadIdx.x * DPT + i;
        s_start[d] = start;
        s_out[d] = __ldg(offsets + T.hist0 + (size_t)d * S.tps) - start;
        start += total[i];
    }
    __syncthreads();
    // the tile in digit order in shared memory
#pragma unroll
    for (int r = 0; r < kSortPerThread; ++r)
        if (base + r * 32 < T.len) {
            const uint32_t d = (uint32_t)(key[r] >> shift) & mask;
            const uint32_t pos = s_start[d] + cnt[w][d] + rank[r];
            s_key[pos] = key[r];
            s_val[pos] = val[r];
        }
    __syncthreads();
    for (int i = threadIdx.x; i < T.len; i += kSortThreads) {
        const K k = s_key[i];
        const uint32_t dst = s_out[(uint32_t)(k >> shift) & mask] + (uint32_t)i;   // n < 2^32
        keys_out[dst] = k;
        vals_out[dst] = s_val[i];
    }
}

// Entries of hist and of the scan's partial sums that sort() needs for one
// segment of n items at 8 bits a digit.
inline long long hist_entries(long long n) { return 256 * ((n + kSortTile - 1) / kSortTile); }
inline long long partial_entries(long long n) { return blsh_scan::tiles_for(hist_entries(n)) + 1; }

// Sorts the segments of keys[0] (and vals[0] alongside) by their bits
// first_bit .. first_bit + key_bits - 1, stably (items equal there keep their
// order), ping-ponging between buffers 0 and 1; *cur receives the index of
// the buffer that holds the result.  implicit: the initial values are the
// items' positions in their segments (vals[0] is not read).  hist: segs << RB
// times tps uint32; partial: a tile sum per 2,048 of them; grand: one uint32.
template <typename K, int RB>
int sort_segments(blsh_ctx *ctx, K *keys[2], uint32_t *vals[2], const Shape &S, int key_bits, int first_bit,
                  bool implicit, uint32_t *hist, uint32_t *partial, uint32_t *grand, cudaStream_t s, int *cur_out) {
    const unsigned tiles = S.segs * S.tps;
    BLSH_CUDA(ctx, cudaFuncSetAttribute(digit_scatter_kernel<K, RB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)scatter_smem<K, RB>()));
    int cur = 0;
    for (int bit = 0; bit < key_bits && tiles > 0; bit += RB) {
        const int shift = first_bit + bit;
        const uint32_t mask = (1u << (key_bits - bit < RB ? key_bits - bit : RB)) - 1u;
        blsh_time_start(ctx, s);
        digit_hist_kernel<K, RB><<<tiles, kSortThreads, 0, s>>>(keys[cur], S, shift, mask, hist);
        BLSH_LAUNCHED(ctx, "digit_hist_kernel");
        const int rc = blsh_scan::run<uint32_t>(ctx, hist, hist, (long long)tiles << RB, partial, grand, s);
        if (rc) return rc;
        blsh_time_start(ctx, s);
        digit_scatter_kernel<K, RB><<<tiles, kSortThreads, scatter_smem<K, RB>(), s>>>(
            keys[cur], bit == 0 && implicit ? nullptr : vals[cur], S, shift, mask, hist, keys[cur ^ 1], vals[cur ^ 1]);
        BLSH_LAUNCHED(ctx, "digit_scatter_kernel");
        cur ^= 1;
    }
    *cur_out = cur;
    return BLSH_OK;
}

// One segment of n 64-bit keys, 8 bits a digit.
inline int sort(blsh_ctx *ctx, unsigned long long *keys[2], uint32_t *vals[2], long long n, int key_bits,
                uint32_t *hist, uint32_t *partial, uint32_t *grand, cudaStream_t s, int *cur_out,
                int first_bit = 0) {
    return sort_segments<unsigned long long, 8>(ctx, keys, vals, shape(n, n > 0 ? 1 : 0), key_bits, first_bit, false,
                                                hist, partial, grand, s, cur_out);
}

}  // namespace blsh_radix
