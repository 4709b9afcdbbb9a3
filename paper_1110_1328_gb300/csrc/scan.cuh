// scan.cuh -- device-wide exclusive prefix sum in three phases (tile sums,
// scan of the tile sums in one CTA, tile scans with their offsets).  Used by
// the banding step for bucket offsets and pair offsets.
#pragma once

#include "common.cuh"

namespace blsh_scan {

constexpr int kThreads = 256;
constexpr int kPerThread = 8;
constexpr int kTile = kThreads * kPerThread;

template <typename T>
__device__ T block_exclusive(T v, T *total) {
    __shared__ T warp_sums[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    T x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[wid] = x;
    __syncthreads();
    if (wid == 0) {
        const int nw = blockDim.x >> 5;
        T s = lane < nw ? warp_sums[lane] : T(0);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const T y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < nw) warp_sums[lane] = s;
    }
    __syncthreads();
    const T before = wid > 0 ? warp_sums[wid - 1] : T(0);
    if (total) *total = warp_sums[(blockDim.x >> 5) - 1];
    const T r = before + x - v;
    __syncthreads();
    return r;
}

template <typename T>
__global__ void __launch_bounds__(kThreads) tile_sums(const T *in, long long n, T *partial) {
    const long long base = (long long)blockIdx.x * kTile;
    T s = 0;
#pragma unroll
    for (int i = 0; i < kPerThread; ++i) {
        const long long p = base + (long long)i * kThreads + threadIdx.x;
        if (p < n) s += in[p];
    }
    T total;
    block_exclusive<T>(s, &total);
    if (threadIdx.x == 0) partial[blockIdx.x] = total;
}

// Exclusive scan of partial[0..m) in place by one CTA; *grand = the sum.
template <typename T>
__global__ void __launch_bounds__(1024) scan_partials(T *partial, long long m, T *grand) {
    __shared__ T carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (long long c0 = 0; c0 < m; c0 += blockDim.x) {
        const long long p = c0 + threadIdx.x;
        const T v = p < m ? partial[p] : T(0);
        T tot;
        const T ex = block_exclusive<T>(v, &tot);
        const T base = carry;
        if (p < m) partial[p] = base + ex;
        __syncthreads();
        if (threadIdx.x == 0) carry = base + tot;
        __syncthreads();
    }
    if (threadIdx.x == 0 && grand) *grand = carry;
}

// out[p] = partial[tile] + exclusive scan within the tile (in may equal out).
template <typename T>
__global__ void __launch_bounds__(kThreads) tile_apply(const T *in, T *out, long long n, const T *partial) {
    const long long base = (long long)blockIdx.x * kTile + (long long)threadIdx.x * kPerThread;
    T v[kPerThread];
    T s = 0;
#pragma unroll
    for (int i = 0; i < kPerThread; ++i) {
        const long long p = base + i;
        v[i] = p < n ? in[p] : T(0);
        s += v[i];
    }
    T ex = block_exclusive<T>(s, nullptr) + partial[blockIdx.x];
#pragma unroll
    for (int i = 0; i < kPerThread; ++i) {
        const long long p = base + i;
        if (p < n) out[p] = ex;
        ex += v[i];
    }
}

// The whole scan in one CTA, eight entries a thread at a time.
template <typename T>
__global__ void __launch_bounds__(1024) scan_small(const T *in, T *out, int n, T *grand) {
    T carry = 0;
    for (int c0 = 0; c0 < n; c0 += 1024 * kPerThread) {
        const int base = c0 + (int)threadIdx.x * kPerThread;
        T v[kPerThread];
        T s = 0;
#pragma unroll
        for (int i = 0; i < kPerThread; ++i) {
            v[i] = base + i < n ? in[base + i] : T(0);
            s += v[i];
        }
        T tot;
        T ex = carry + block_exclusive<T>(s, &tot);
#pragma unroll
        for (int i = 0; i < kPerThread; ++i) {
            if (base + i < n) out[base + i] = ex;
            ex += v[i];
        }
        carry += tot;
    }
    if (threadIdx.x == 0 && grand) *grand = carry;
}

// Up to this many entries one CTA scans in less time than three launches take:
// 8,192 entries of 4 bytes 8.3 us against 12.3, of 8 bytes 10.3 / 13.4; 16,384
// entries 14.5 / 12.3 and 16.5 / 13.4, 32,768 26.7 / 12.3 and 30.8 / 14.4.
constexpr long long kSmallScan = 8192;

inline long long tiles_for(long long n) { return (n + kTile - 1) / kTile; }

// Exclusive scan of in[0..n) into out (may alias); *grand (device) = total.
// `partial` needs tiles_for(n) elements.  *launches (if given) = the kernels launched.
template <typename T>
cudaError_t exclusive_scan(const T *in, T *out, long long n, T *partial, T *grand, cudaStream_t s,
                           int *launches = nullptr) {
    const long long tiles = tiles_for(n);
    if (launches) *launches = tiles == 0 ? 0 : n <= kSmallScan ? 1 : 3;
    if (tiles == 0) return cudaMemsetAsync(grand, 0, sizeof(T), s);
    if (n <= kSmallScan) {
        scan_small<T><<<1, 1024, 0, s>>>(in, out, (int)n, grand);
        return cudaGetLastError();
    }
    tile_sums<T><<<(unsigned)tiles, kThreads, 0, s>>>(in, n, partial);
    scan_partials<T><<<1, 1024, 0, s>>>(partial, tiles, grand);
    tile_apply<T><<<(unsigned)tiles, kThreads, 0, s>>>(in, out, n, partial);
    return cudaGetLastError();
}

// exclusive_scan with the context's launch count, timing record and status.
template <typename T>
int run(blsh_ctx *ctx, const T *in, T *out, long long n, T *partial, T *grand, cudaStream_t s) {
    int launches = 0;
    blsh_time_start(ctx, s);
    BLSH_CUDA(ctx, exclusive_scan<T>(in, out, n, partial, grand, s, &launches));
    ctx->launches.fetch_add(launches, std::memory_order_relaxed);
    blsh_time_stop(ctx, "exclusive scan");
    return BLSH_OK;
}

}  // namespace blsh_scan
