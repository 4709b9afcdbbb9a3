// compact.cu -- the output set O of Algorithms 1 and 2: a stable compaction
// of the retained pair indices.
//
// Few statuses take one launch (compact_few).  Otherwise a fixed grid of C CTAs
// splits [0, P) into C contiguous ranges, read 16 statuses at a time.  Pass 1
// counts the kept items of each range (1e9 statuses: 0.30 ms at one load in
// flight a thread, 0.19 with eight; pass 2 0.52 and 0.39); pass 2 gives each CTA the sum of the
// counts of the ranges before it and writes its range's indices in order,
// one tile at a time with a block-wide prefix sum.  The count array (C
// entries) lives in the context's scratch area.
#include "common.cuh"
#include "scan.cuh"

namespace {

constexpr int kThreads = 256;
constexpr int kPer = 16;
constexpr int kTile = kThreads * kPer;
constexpr int kBatch = 8;   // tiles whose loads are in flight together

__device__ __forceinline__ bool kept(uint8_t st, uint32_t mask) { return st < 32 && ((mask >> st) & 1u); }

__device__ __forceinline__ long long resolve_p(long long P, const long long *P_dev) {
    if (!P_dev) return P;
    const long long pd = *P_dev;
    return pd < 0 ? 0 : (pd < P ? pd : P);
}

// The status array may start anywhere: `off` is its address modulo 16, and
// ranges and tiles begin at multiples of 16 of the index plus off, so that every
// 16 statuses but the first ones are one 16-byte load.
// CTA b owns [lo, hi), about P b / C on; the first begins at -off (statuses
// below 0 are none).
__device__ __forceinline__ void cta_range(long long P, int off, long long &lo, long long &hi) {
    lo = ((P * blockIdx.x / gridDim.x + off) & ~15ll) - off;
    hi = blockIdx.x + 1 == gridDim.x ? P : ((P * (blockIdx.x + 1) / gridDim.x + off) & ~15ll) - off;
}

// Bit i: status i (a byte of v) is kept (a shift past 31 gives 0): about four
// operations a status, whatever the mask.
__device__ __forceinline__ uint32_t kept4(uint32_t v, uint32_t mask) {
    uint32_t r = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        uint32_t k;
        asm("shr.u32 %0, %1, %2;" : "=r"(k) : "r"(mask), "r"((v >> (8 * i)) & 0xffu));   // (clamped at 32)
        r |= (k & 1u) << i;
    }
    return r;
}

// Bit i of the result: status i of v is kept.  One or two kept statuses are
// matched in all 16 bytes at once, about 45 operations each; more cost what
// kept4 does.
__device__ __forceinline__ uint32_t kept16(uint4 v, uint32_t mask) {
    if (__popc(mask) > 2) return kept4(v.x, mask) | kept4(v.y, mask) << 4 | kept4(v.z, mask) << 8 | kept4(v.w, mask) << 12;
    uint32_t bits = 0;
    for (uint32_t m = mask; m; m &= m - 1) bits |= blsh_eq16(v, (uint32_t)(__ffs(m) - 1));
    return bits;
}

// bits[u], bit i: status q0 + u step + i is kept (and lies below hi).  The U
// loads come first, without a branch between them, so that all are in flight:
// with each inside its own loop over the kept statuses a thread had one, and
// 1e9 statuses were read at 3.3 TB/s.
template <int U>
__device__ __forceinline__ void kept_tiles(const uint8_t *status, long long q0, long long step, long long hi,
                                           uint32_t mask, uint32_t (&bits)[U]) {
    if (q0 >= 0 && q0 + (U - 1) * step + 16 <= hi) {
        uint4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = __ldg(reinterpret_cast<const uint4 *>(status + q0 + u * step));
#pragma unroll
        for (int u = 0; u < U; ++u) bits[u] = kept16(v[u], mask);
    } else {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long long q = q0 + u * step;
            bits[u] = 0;
            if (q >= hi) continue;
            if (q >= 0 && q + 16 <= hi) {
                bits[u] = kept16(__ldg(reinterpret_cast<const uint4 *>(status + q)), mask);
            } else {
                for (int i = 0; i < 16; ++i)
                    if (q + i >= 0 && q + i < hi) bits[u] |= (uint32_t)kept(status[q + i], mask) << i;
            }
        }
    }
}

// Up to kFew statuses: one launch.  CTA b writes the indices of 4,096 statuses,
// in order from shared memory so that the stores are coalesced, and counts the
// kept ones before them itself (at most 128 KB, from L2, every load in flight)
// instead of waiting for a count pass: the second launch costs more.  Those
// past the device's count end at once.  (One CTA for all of them wrote its
// indices a lane each: 131,072 statuses, all kept, 79 us, 12.0 in two launches;
// 8.7 here.  200 in use: 12.6 in two launches, 8.7 here.)
constexpr int kFewThreads = 1024, kFewTile = 4 * kFewThreads, kFewLoads = 8;
constexpr long long kFew = (long long)kFewThreads * kPer * kFewLoads;
__global__ void __launch_bounds__(kFewThreads) compact_few(const uint8_t *status, long long P_cap,
                                                           const long long *P_dev, uint32_t mask, int off,
                                                           int64_t *out, long long cap, long long *n_out,
                                                           blsh_dev_scratch *scratch) {
    __shared__ int s_before[32], s_own[32];
    __shared__ uint16_t s_list[kFewTile];
    const int P = (int)resolve_p(P_cap, P_dev), lo = (int)blockIdx.x * kFewTile - off;   // (the first begins at -off)
    if (lo >= P && blockIdx.x > 0) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, t = threadIdx.x;
    auto by_one = [&](int q, int n) {   // statuses q .. q + n - 1, those that are there
        uint32_t b = 0;
        for (int i = 0; i < n; ++i)
            if (q + i >= 0 && q + i < P) b |= (uint32_t)kept(status[q + i], mask) << i;
        return b;
    };
    uint4 v[kFewLoads];   // the statuses before this CTA's, chunks of 16 from -off on
#pragma unroll
    for (int u = 0; u < kFewLoads; ++u) {
        const int q = (t + u * kFewThreads) * kPer - off;
        v[u] = q >= 0 && q < lo ? __ldg(reinterpret_cast<const uint4 *>(status + q)) : make_uint4(~0u, ~0u, ~0u, ~0u);
    }
    const int q = lo + 4 * t;   // its own, four a thread
    const uint32_t own = q >= 0 && q + 4 <= P ? kept4(__ldg(reinterpret_cast<const uint32_t *>(status + q)), mask)
                                              : by_one(q, 4);
    int before = t == 0 && off && lo > 0 ? __popc(by_one(-off, kPer)) : 0;   // the first chunk, where it is not whole
#pragma unroll
    for (int u = 0; u < kFewLoads; ++u)
        if (u * kFewThreads * kPer < lo + off) before += __popc(kept16(v[u], mask));   // (the CTA has any there)
    before = __reduce_add_sync(0xffffffffu, before);
    const int c = __popc(own);
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) {
        s_before[warp] = before;
        s_own[warp] = incl;
    }
    __syncthreads();
    const int base = __reduce_add_sync(0xffffffffu, s_before[lane]);
    const int total = __reduce_add_sync(0xffffffffu, s_own[lane]);
    int at = incl - c + __reduce_add_sync(0xffffffffu, lane < warp ? s_own[lane] : 0);
    for (uint32_t b = own; b; b &= b - 1) s_list[at++] = (uint16_t)(4 * t + __ffs(b) - 1);
    __syncthreads();
    for (int i = t; i < total; i += kFewThreads)
        if ((long long)base + i < cap) out[base + i] = lo + s_list[i];
    if (lo + kFewTile >= P && t == 0) {   // the last of them
        const long long n = (long long)base + total;
        *n_out = n;
        if (n > cap) blsh_dev_error(scratch, BLSH_ETRUNC, 1, (unsigned long long)(n - cap));
    }
}

__global__ void __launch_bounds__(kThreads) compact_count(const uint8_t *status, long long P_cap,
                                                          const long long *P_dev, uint32_t mask, int off,
                                                          blsh_dev_scratch *scratch) {
    const long long P = resolve_p(P_cap, P_dev);
    long long lo, hi;
    cta_range(P, off, lo, hi);
    long long c = 0;
    for (long long q0 = lo + 16ll * threadIdx.x; q0 < hi; q0 += (long long)kBatch * kTile) {
        uint32_t bits[kBatch];
        kept_tiles<kBatch>(status, q0, kTile, hi, mask, bits);
#pragma unroll
        for (int u = 0; u < kBatch; ++u) c += __popc(bits[u]);
    }
    long long total;
    blsh_scan::block_exclusive<long long>(c, &total);
    if (threadIdx.x == 0) scratch->cta_counts[blockIdx.x] = total;
}

// Writes the indices of [lo, hi) from out[base] on and returns the place after
// them.  kBatch tiles at a time: their loads are issued together, then each tile
// gets its block-wide prefix sum and its indices leave in order.  STAGED: a
// warp's from shared memory, 32 at a time, else by the lanes that hold them.
template <bool STAGED>
__device__ __forceinline__ long long write_range(const uint8_t *status, long long lo, long long hi, uint32_t mask,
                                                 long long base, int64_t *out, long long cap, uint16_t *list) {
    for (long long t0 = lo; t0 < hi; t0 += (long long)kBatch * kTile) {
        uint32_t bits[kBatch];
        kept_tiles<kBatch>(status, t0 + (long long)threadIdx.x * kPer, kTile, hi, mask, bits);
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            if (t0 + (long long)u * kTile >= hi) break;      // uniform across the CTA
            const long long q0 = t0 + (long long)u * kTile + (long long)threadIdx.x * kPer;
            long long tile_total;
            long long o = base + blsh_scan::block_exclusive<long long>((long long)__popc(bits[u]), &tile_total);
            if constexpr (STAGED) {
                const int lane = threadIdx.x & 31;
                const long long first = __shfl_sync(0xffffffffu, o, 0);
                int at = (int)(o - first);
                for (uint32_t b = bits[u]; b; b &= b - 1) list[at++] = (uint16_t)(kPer * lane + __ffs(b) - 1);
                const int n = __shfl_sync(0xffffffffu, at, 31);
                __syncwarp();
                for (int i = lane; i < n; i += 32)
                    if (first + i < cap) out[first + i] = q0 - kPer * lane + list[i];
                __syncwarp();
            } else {
                for (uint32_t b = bits[u]; b; b &= b - 1) {
                    if (o < cap) out[o] = q0 + __ffs(b) - 1;
                    ++o;
                }
            }
            base += tile_total;
        }
    }
    return base;
}

// A CTA stages its indices where more than a kFewKept-th of its statuses are kept
// (1e8 statuses, all kept, a lane writing its own 16: 894 us, 190 here; 30% 124,
// 110).  The two loops are apart because one with both forms, chosen warp by warp
// or tile by tile, took longer where few are kept (1e9 statuses: 464 and 454 us,
// 442 here).
constexpr int kFewKept = 4;
__global__ void __launch_bounds__(kThreads) compact_write(const uint8_t *status, long long P_cap,
                                                          const long long *P_dev, uint32_t mask, int off,
                                                          int64_t *out, long long cap, long long *n_out,
                                                          blsh_dev_scratch *scratch) {
    __shared__ long long s_base;
    __shared__ uint16_t s_list[kThreads / 32][32 * kPer];
    const long long P = resolve_p(P_cap, P_dev);
    long long lo, hi;
    cta_range(P, off, lo, hi);
    long long before = 0;
    for (int c = threadIdx.x; c < (int)blockIdx.x; c += kThreads) before += scratch->cta_counts[c];
    long long tot;
    blsh_scan::block_exclusive<long long>(before, &tot);
    if (threadIdx.x == 0) s_base = tot;
    __syncthreads();
    long long base = s_base;
    base = scratch->cta_counts[blockIdx.x] > (unsigned long long)(hi > lo ? hi - lo : 0) / kFewKept
               ? write_range<true>(status, lo, hi, mask, base, out, cap, s_list[threadIdx.x >> 5])
               : write_range<false>(status, lo, hi, mask, base, out, cap, nullptr);
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
        *n_out = base;
        if (base > cap) blsh_dev_error(scratch, BLSH_ETRUNC, 1, (unsigned long long)(base - cap));
    }
}

}  // namespace

extern "C" int blsh_compact(blsh_ctx *ctx, const uint8_t *status, int64_t P, const int64_t *P_dev,
                            uint32_t keep_mask, int64_t *out_idx, int64_t cap, int64_t *n_out, void *stream) {
    if (!ctx) return BLSH_EINVAL;
    if (!n_out || (P > 0 && !status) || (cap > 0 && !out_idx))
        return blsh_fail(ctx, BLSH_EINVAL, "status and n_out required");
    if (P < 0 || cap < 0) return blsh_fail(ctx, BLSH_EINVAL, "bad P or cap");
    if (!blsh_aligned(out_idx, 8) || !blsh_aligned(n_out, 8) || !blsh_aligned(P_dev, 8))
        return blsh_fail(ctx, BLSH_EINVAL, "misaligned pointer");
    blsh_device_guard g(ctx->device);
    cudaStream_t s = blsh_stream(stream);
    long long ctas = (P + kTile - 1) / kTile;
    const long long most = (long long)ctx->sm_count * 4 < BLSH_COMPACT_MAX_CTAS ? (long long)ctx->sm_count * 4
                                                                                 : BLSH_COMPACT_MAX_CTAS;
    if (ctas > most) ctas = most;
    if (ctas < 1) ctas = 1;
    const int off = (int)((uintptr_t)status & 15);
    if (P <= kFew) {
        const unsigned few = (unsigned)((P + off + kFewTile - 1) / kFewTile);
        blsh_time_start(ctx, s);
        compact_few<<<few > 0 ? few : 1u, kFewThreads, 0, s>>>(status, P, (const long long *)P_dev, keep_mask, off,
                                                               out_idx, cap, (long long *)n_out, ctx->scratch);
        BLSH_LAUNCHED(ctx, "compact_few");
        return BLSH_OK;
    }
    blsh_time_start(ctx, s);
    compact_count<<<(unsigned)ctas, kThreads, 0, s>>>(status, P, (const long long *)P_dev, keep_mask, off,
                                                      ctx->scratch);
    BLSH_LAUNCHED(ctx, "compact_count");
    blsh_time_start(ctx, s);
    compact_write<<<(unsigned)ctas, kThreads, 0, s>>>(status, P, (const long long *)P_dev, keep_mask, off, out_idx,
                                                      cap, (long long *)n_out, ctx->scratch);
    BLSH_LAUNCHED(ctx, "compact_write");
    return BLSH_OK;
}
