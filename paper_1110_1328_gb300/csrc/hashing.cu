// hashing.cu -- the signature producers: minhash (Section 4.1, "LSH family")
// and sign random projections of sparse rows (Section 4.2, "LSH family").
#include <stddef.h>

#include <type_traits>

#include "common.cuh"

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr uint32_t kP31 = 0x7fffffffu;   // 2^31 - 1

// v mod (2^31 - 1) for any 32-bit v.
__device__ __forceinline__ uint32_t mod_p31(uint32_t v) {
    const uint32_t f = (v & kP31) + (v >> 31);   // at most 2^31
    return f >= kP31 ? f - kP31 : f;
}

// The running minimum of (a x + b) mod p, p = 2^31 - 1, for a, b, x < p, given
// a2 = 2a and b2 = 2b: with v = a x + b < p (p - 1) + p, the high word of 2v is
// v >> 31 < p and the low word is 2 (v mod 2^31), so r = high + low / 2 is
// congruent to v and below 2p: the residue is r or r - p, and where r < p the
// difference wraps to a larger number, so the three-way minimum takes the
// right one.  Four instructions (multiply-add to 64 bits, shift-and-add,
// subtract, minimum) against about twelve for folding twice and subtracting
// under a test; the integer pipe is what this kernel waits for.
__device__ __forceinline__ uint32_t min_hash31(uint32_t mn, uint32_t a2, uint32_t b2, uint32_t x) {
    const unsigned long long v2 = (unsigned long long)a2 * x + b2;
    const uint32_t r = (uint32_t)(v2 >> 32) + ((uint32_t)v2 >> 1);
    return __vimin3_u32(mn, r, r - kP31);
}

// Minima over elements [s, e) of the hashes whose a2, b2 the lanes hold:
// elements are read 32 at a time, one per lane, and broadcast; a partial
// block repeats its last element (a minimum does not change) up to a multiple
// of four, so that the loop runs four elements at a time.
template <int HPL>
__device__ __forceinline__ void min_hash_run(const uint32_t *__restrict__ indices, long long s, long long e,
                                             const uint32_t (&a2)[HPL], const uint32_t (&b2)[HPL],
                                             uint32_t (&mn)[HPL]) {
    const int lane = threadIdx.x & 31;
    for (long long e0 = s; e0 < e; e0 += 32) {
        const int cnt = (int)min(32ll, e - e0);
        const uint32_t mine = mod_p31(__ldg(indices + e0 + min(lane, cnt - 1)));
        for (int l = 0; l < cnt; l += 4) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t x = __shfl_sync(kFull, mine, l + q);   // lanes past cnt hold the last element
#pragma unroll
                for (int u = 0; u < HPL; ++u) mn[u] = min_hash31(mn[u], a2[u], b2[u], x);
            }
        }
    }
}

// One warp per (set, tile of 32 HPL hashes): lane l owns hashes l, l + 32, ...
// of a tile and keeps their running minima in registers.  A warp
// alone takes about 46 ns an element, so sets longer than kBigSet are listed
// for minhash_big_kernel: the degrees of a
// graph follow a power law, and a set of 150,000 elements would hold up one
// warp for milliseconds.
//
// Two lists, an entry a set: sets of more than kHubSet elements in one of their
// own (2^20 of them), so that however many others there are (2^23 in the other
// list) a hub is never one warp's work while a warp's worth of others is.  An
// entry holds the set and the number of 32-element blocks listed before it; the
// list's counter holds both numbers, entries above the blocks, so that one
// atomic gives an entry its place and its blocks' place.  The row of a listed
// set starts at the identity of the minimum; that of a set past its list's end
// at a value that no hash takes (its first words), by which minhash_big_kernel
// finds it: those sets are a warp's work each.
// (Entries of 256 elements and a tile on one list of 2^20: 1.5e6 sets of 300
// and then 20 hubs of 1e6 took 109 ms, the hubs a warp each; 25 here.)
//
// 1e6 neighbour lists (mean 27) x 256 hashes, both kernels: 4.77 ms with
// twelve instructions a hash and long sets spread over whole CTAs, 1.56 now
// (4.4e12 hashes/s; 4.9e12 where every set has 64 elements or more, the
// rate of the 64-bit multiply-add and the four others at this mix).
constexpr long long kBigSet = 256;
constexpr long long kHubSet = 2048;
constexpr int kListShift = 36;          // 2^36 blocks and 2^28 entries: more than 280 GB of elements
constexpr unsigned kPartBlocks = 4;     // blocks of a list a warp takes, at least
constexpr uint32_t kListed = 0xffffffffu, kUnlisted = 0xfffffffeu;

struct LongSets {
    uint2 *set, *hub;                   // [BLSH_LITE_QUEUE_CAP], [BLSH_RECHECK_CAP]
    unsigned long long *n_set, *n_hub;  // entries << kListShift | blocks
    unsigned long long *next;           // [2]: the next part of the hubs, of the others
};

// Lists a long set [s, e) (one warp); false if its list is full.
__device__ __forceinline__ bool list_long_set(const LongSets &L, long long i, long long s, long long e) {
    const bool is_hub = e - s > kHubSet;
    unsigned long long before = 0;
    if ((threadIdx.x & 31) == 0)
        before = atomicAdd(is_hub ? L.n_hub : L.n_set, 1ull << kListShift | (unsigned long long)(e - s + 31) >> 5);
    before = __shfl_sync(kFull, before, 0);
    const unsigned long long slot = before >> kListShift;
    if (slot >= (is_hub ? BLSH_RECHECK_CAP : BLSH_LITE_QUEUE_CAP)) return false;
    if ((threadIdx.x & 31) == 0) (is_hub ? L.hub : L.set)[slot] = make_uint2((uint32_t)i, (uint32_t)before);   // (< 2^32 blocks)
    return true;
}

// The coefficients of the lane's hashes in a tile.
template <int HPL>
__device__ __forceinline__ void load_coeffs(const uint32_t *__restrict__ A, const uint32_t *__restrict__ B,
                                            unsigned tile, uint32_t (&a2)[HPL], uint32_t (&b2)[HPL]) {
    const size_t h0 = (size_t)tile * 32 * HPL + (threadIdx.x & 31);
#pragma unroll
    for (int u = 0; u < HPL; ++u) {
        a2[u] = 2u * mod_p31(__ldg(A + h0 + 32 * u));
        b2[u] = 2u * mod_p31(__ldg(B + h0 + 32 * u));
    }
}

// (The bounds choose the compiler's schedule: 1e6 sets of 27 x 256 hashes 1.48 ms,
// 1.53 without; 3e5 of 100 x 128 0.84, 0.86 without, 0.85 with four CTAs.)
template <int HPL>
__global__ void __launch_bounds__(256, HPL == 4 ? 5 : 4) minhash_kernel(
    const int64_t *__restrict__ indptr, const uint32_t *__restrict__ indices, long long N, int n_hashes,
    const uint32_t *__restrict__ A, const uint32_t *__restrict__ B, uint32_t *__restrict__ sig, const LongSets L) {
    const int lane = threadIdx.x & 31;
    const unsigned tiles = (unsigned)n_hashes / (32u * HPL);
    const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
    for (unsigned tile = blockIdx.y; tile < tiles; tile += gridDim.y) {
        const int h0 = (int)tile * 32 * HPL + lane;
        uint32_t a2[HPL], b2[HPL];
        load_coeffs<HPL>(A, B, tile, a2, b2);
        for (long long i = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < N; i += warps) {
            const long long s = __ldg(indptr + i), e = __ldg(indptr + i + 1);
            uint32_t mn[HPL];
#pragma unroll
            for (int u = 0; u < HPL; ++u) mn[u] = kListed;
            if (e - s <= kBigSet) {
                min_hash_run<HPL>(indices, s, e, a2, b2, mn);
            } else if (tile == 0 && !list_long_set(L, i, s, e)) {   // (all its tiles are listed at once)
#pragma unroll
                for (int u = 0; u < HPL; ++u) mn[u] = kUnlisted;
            }
#pragma unroll
            for (int u = 0; u < HPL; ++u) sig[(size_t)i * n_hashes + h0 + 32 * u] = mn[u];
        }
    }
}

// The same for few sets: a CTA per (set, tile), its eight warps taking an
// eighth of the elements each, their minima joined in shared memory.  (There
// are fewer sets than the list of hubs holds.)
template <int HPL>
__global__ void __launch_bounds__(256) minhash_cta_kernel(const int64_t *__restrict__ indptr,
                                                          const uint32_t *__restrict__ indices, int n_hashes,
                                                          const uint32_t *__restrict__ A,
                                                          const uint32_t *__restrict__ B, uint32_t *__restrict__ sig,
                                                          const LongSets L) {
    __shared__ uint32_t red[8][32 * HPL];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long i = blockIdx.x;
    const long long s = __ldg(indptr + i), e = __ldg(indptr + i + 1);
    if (e - s > kHubSet) {
        if (blockIdx.y == 0) {
            if (warp == 0) list_long_set(L, i, s, e);
            for (int k = threadIdx.x; k < n_hashes; k += 256) sig[(size_t)i * n_hashes + k] = kListed;
        }
        return;
    }
    uint32_t a2[HPL], b2[HPL], mn[HPL];
    load_coeffs<HPL>(A, B, blockIdx.y, a2, b2);
#pragma unroll
    for (int u = 0; u < HPL; ++u) mn[u] = 0xffffffffu;
    const long long piece = (e - s + 7) >> 3;
    const long long s0 = s + warp * piece, e0 = s0 + piece < e ? s0 + piece : e;
    min_hash_run<HPL>(indices, s0, e0, a2, b2, mn);
#pragma unroll
    for (int u = 0; u < HPL; ++u) red[warp][32 * u + lane] = mn[u];
    __syncthreads();
    if (threadIdx.x < 32 * HPL) {
        uint32_t m = red[0][threadIdx.x];
#pragma unroll
        for (int w = 1; w < 8; ++w) m = min(m, red[w][threadIdx.x]);
        sig[(size_t)i * n_hashes + (size_t)blockIdx.y * 32 * HPL + threadIdx.x] = m;
    }
}

// The listed sets: a list's blocks are cut into equal parts, about four a warp
// over all tiles, whatever sets they lie in, and handed out from a counter; a
// part's minima of a set meet in the set's row
// in global memory (atomicMin: the minimum does not depend on the order).
template <int HPL>
__device__ __forceinline__ void hash_listed(const uint2 *list, unsigned long long count, unsigned long long cap,
                                            unsigned long long *next,
                                            const int64_t *__restrict__ indptr, const uint32_t *__restrict__ indices,
                                            int n_hashes, const uint32_t *__restrict__ A,
                                            const uint32_t *__restrict__ B, uint32_t *__restrict__ sig) {
    const int lane = threadIdx.x & 31;
    const unsigned long long entries = count >> kListShift;
    if (entries == 0) return;
    const unsigned n = (unsigned)(entries < cap ? entries : cap);
    unsigned total = (unsigned)count;                  // (< 2^32 blocks)
    if (entries > cap) {
        const uint2 last = list[n - 1];
        total = last.y + (unsigned)((__ldg(indptr + last.x + 1) - __ldg(indptr + last.x) + 31) >> 5);
    }
    const unsigned tiles = (unsigned)n_hashes / (32u * HPL), warps = gridDim.x * (blockDim.x >> 5);
    const unsigned per_tile = 4 * warps / tiles > 0 ? 4 * warps / tiles : 1u;
    unsigned part = (total - 1) / per_tile + 1;
    if (part < kPartBlocks) part = kPartBlocks;
    const unsigned parts = (total - 1) / part + 1;     // parts tiles <= 4 warps, unless the tiles alone are more
    for (;;) {
        unsigned u = 0;
        if (lane == 0) u = (unsigned)atomicAdd(next, 1ull);
        u = __shfl_sync(kFull, u, 0);
        if (u >= parts * tiles) break;
        const unsigned tile = u / parts;
        unsigned b = (u - tile * parts) * part;        // the next block
        const unsigned end = total - b > part ? b + part : total;
        unsigned q = 0, hi = n;                        // its set: the last that starts at or before it
        while (hi - q > 1) {
            const unsigned mid = q + (hi - q) / 2;
            if (list[mid].y <= b) q = mid; else hi = mid;
        }
        uint32_t a2[HPL], b2[HPL];
        load_coeffs<HPL>(A, B, tile, a2, b2);
        for (; b < end; ++q) {
            const uint2 ent = list[q];
            long long s = __ldg(indptr + ent.x), e = __ldg(indptr + ent.x + 1);
            const unsigned next = ent.y + (unsigned)((e - s + 31) >> 5);   // the set's last block, and one
            const unsigned to = next < end ? next : end;
            if (next > end) e = s + 32ll * (end - ent.y);
            s += 32ll * (b - ent.y);
            b = to;
            uint32_t mn[HPL];
#pragma unroll
            for (int v = 0; v < HPL; ++v) mn[v] = 0xffffffffu;
            min_hash_run<HPL>(indices, s, e, a2, b2, mn);
            uint32_t *row = sig + (size_t)ent.x * n_hashes + (size_t)tile * 32 * HPL + lane;
#pragma unroll
            for (int v = 0; v < HPL; ++v) atomicMin(row + 32 * v, mn[v]);
        }
    }
}

template <int HPL>
__global__ void __launch_bounds__(256) minhash_big_kernel(const int64_t *__restrict__ indptr,
                                                          const uint32_t *__restrict__ indices, long long N,
                                                          int n_hashes, const uint32_t *__restrict__ A,
                                                          const uint32_t *__restrict__ B,
                                                          uint32_t *__restrict__ sig, const LongSets L) {
    // one copy of the code for both lists: hubs first
#pragma unroll 1
    for (int set = 0; set < 2; ++set)
        hash_listed<HPL>(set ? L.set : L.hub, set ? *L.n_set : *L.n_hub, set ? BLSH_LITE_QUEUE_CAP : BLSH_RECHECK_CAP,
                         L.next + set, indptr, indices, n_hashes, A, B, sig);
    if (*L.n_hub >> kListShift <= BLSH_RECHECK_CAP && *L.n_set >> kListShift <= BLSH_LITE_QUEUE_CAP) return;
    const unsigned tiles = (unsigned)n_hashes / (32u * HPL);
    const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long i = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < N; i += warps) {
        const long long s = __ldg(indptr + i), e = __ldg(indptr + i + 1);
        uint32_t *row = sig + (size_t)i * n_hashes + (threadIdx.x & 31);
        if (e - s <= kBigSet || sig[(size_t)i * n_hashes] != kUnlisted) continue;
        for (unsigned tile = 0; tile < tiles; ++tile) {
            uint32_t a2[HPL], b2[HPL], mn[HPL];
            load_coeffs<HPL>(A, B, tile, a2, b2);
#pragma unroll
            for (int u = 0; u < HPL; ++u) mn[u] = 0xffffffffu;
            min_hash_run<HPL>(indices, s, e, a2, b2, mn);
#pragma unroll
            for (int u = 0; u < HPL; ++u) row[(size_t)tile * 32 * HPL + 32 * u] = mn[u];
        }
    }
}

// Sign random projections of sparse rows.  One CTA per row (grid-stride);
// thread t owns bits t, t+T, ..., so that the threads of a warp read 128
// contiguous bytes of a row of R and a warp ballot of one of its bits forms
// one signature word.  Sums are FP32 with fused multiply-adds in row order;
// next to each sum the thread keeps sum |v r|.  Recursive summation of n
// exact products has error at most (n-1) u sum|v r| (u = 2^-24); a sum whose
// magnitude exceeds 1.25 n u sum|v r| + n 2^-149 has the sign of the exact
// sum (and of the FP64 row-order sum, whose error is 2^29 times smaller).
// Otherwise the thread recomputes the sum in FP64 in row order, which
// reproduces that FP64 sum bit for bit (products of floats are exact in FP64,
// so one rounding per addition with or without fusion).
// Entry (i) of R as FP64: a float, or a two-byte code q read back as
// q 2^-12 - 8 (Section 4.3), which is exact in FP64 (and in FP32).
__device__ __forceinline__ double r_fp64(const float *R, size_t i) { return (double)__ldg(R + i); }
__device__ __forceinline__ double r_fp64(const uint16_t *R, size_t i) {
    return (double)__ldg(R + i) * (1.0 / 4096.0) - 8.0;
}
__device__ __forceinline__ float r_fp32(const float *R, size_t i) { return __ldg(R + i); }
__device__ __forceinline__ float r_fp32(const uint16_t *R, size_t i) {
    return __fmaf_rn((float)__ldg(R + i), 1.0f / 4096.0f, -8.0f);
}

constexpr int kSrpMaxPerThread = 16;
constexpr int kSrpBatch = 8;        // gathers issued together
constexpr int kSrpChunk = 256;

template <typename RT>
__global__ void __launch_bounds__(256) srp_sparse_kernel(const int64_t *__restrict__ indptr,
                                                         const uint32_t *__restrict__ indices,
                                                         const float *__restrict__ values, long long N,
                                                         const RT *__restrict__ R, long long dim, int bits,
                                                         int per_thread,
                                                         uint32_t *__restrict__ sig, blsh_dev_scratch *scratch) {
    __shared__ uint32_t s_idx[kSrpChunk];
    __shared__ float s_val[kSrpChunk];
    const int T = blockDim.x;
    const int t = threadIdx.x;
    const int words = bits >> 5;
    unsigned long long rechecked = 0, zeros = 0;
    for (long long row = blockIdx.x; row < N; row += gridDim.x) {
        const long long s = __ldg(indptr + row), e = __ldg(indptr + row + 1);
        float acc[kSrpMaxPerThread], mag[kSrpMaxPerThread];
#pragma unroll
        for (int u = 0; u < kSrpMaxPerThread; ++u) acc[u] = mag[u] = 0.0f;
        for (long long c0 = s; c0 < e; c0 += kSrpChunk) {
            const int cnt = (int)min((long long)kSrpChunk, e - c0);
            __syncthreads();
            for (int i = t; i < cnt; i += T) {
                uint32_t ix = __ldg(indices + c0 + i);
                float v = __ldg(values + c0 + i);
                if (ix >= dim) {   // malformed row: record it, contribute nothing
                    blsh_dev_error(scratch, BLSH_ERANGE, 0, 1ull);
                    ix = 0;
                    v = 0.0f;
                }
                s_idx[i] = ix;
                s_val[i] = v;
            }
            __syncthreads();
            for (int i = 0; i < cnt; ++i) {
                const float v = s_val[i];
                const RT *Rrow = R + (size_t)s_idx[i] * bits + t;
#pragma unroll
                for (int u = 0; u < kSrpMaxPerThread; ++u) {
                    if (u < per_thread) {
                        const float r = r_fp32(Rrow, (size_t)u * T);
                        acc[u] = __fmaf_rn(v, r, acc[u]);
                        mag[u] = __fmaf_rn(fabsf(v), fabsf(r), mag[u]);
                    }
                }
            }
        }
        const float n = (float)(int)(e - s < (1ll << 30) ? e - s : (1ll << 30));   // 32-bit conversion
        const bool long_row = n * 5.9604644775390625e-8f > 0.05f;   // the 1.25 slack needs n u <= 0.05
        const int w = t >> 5;
#pragma unroll
        for (int u = 0; u < kSrpMaxPerThread; ++u) {
            if (u < per_thread) {
                const float bound = 1.25f * n * 5.9604644775390625e-8f * mag[u] + n * 1.4e-45f;
                bool bit;
                if (!long_row && fabsf(acc[u]) > bound) {
                    bit = acc[u] >= 0.0f;
                } else {
                    double d = 0.0;
                    for (long long k = s; k < e; ++k) {
                        const uint32_t ix = __ldg(indices + k);
                        if (ix < dim) d += (double)__ldg(values + k) * r_fp64(R, (size_t)ix * bits + t + u * T);
                    }
                    bit = d >= 0.0;
                    ++rechecked;
                    zeros += d == 0.0;
                }
                const unsigned word = __ballot_sync(kFull, bit);
                if ((t & 31) == 0) sig[(size_t)row * words + w + u * (T >> 5)] = word;
            }
        }
    }
    if (rechecked) atomicAdd(&scratch->counters[2], rechecked);
    if (zeros) atomicAdd(&scratch->counters[3], zeros);
}


// The FP64 row-order sum of row [s, e) against column j of R, as the oracle
// forms it (rare: only signs the FP32 bound cannot decide).  Kept out of line
// so the hot accumulation loop keeps its registers.
template <typename RT>
__device__ __noinline__ double srp_recheck_fp64(const uint32_t *__restrict__ indices,
                                                const float *__restrict__ values, long long s, long long e,
                                                const RT *__restrict__ R, long long dim, int bits, int j) {
    double d = 0.0;
    for (long long k = s; k < e; ++k) {
        const uint32_t ix = __ldg(indices + k);
        if (ix < dim) d += (double)__ldg(values + k) * r_fp64(R, (size_t)ix * bits + j);
    }
    return d;
}

// The two codes of a 32-bit word as the pair (2^23 + low code, 2^23 + high
// code): each code's bits placed under the exponent of 2^23.
__device__ __forceinline__ unsigned long long f2_codes(uint32_t w) {
    return f2_pack(__int_as_float((int)__byte_perm(w, 0x4b00u, 0x5410)),
                   __int_as_float((int)__byte_perm(w, 0x4b00u, 0x5432)));
}

// The same computation when bits is a multiple of 128 and R is aligned for it:
// a warp per (row, piece of 32 CPL columns), a lane owning CPL neighbouring
// columns -- 16 bytes of a row of R a load (four floats, or eight two-byte
// codes of Section 4.3; four codes where the columns are no multiple of 256 or
// R lies on 8 bytes only).
//
// A grab of G rows comes from a counter: row lengths follow a power law, and a
// fixed share per warp left most of the GPU idle behind the longest rows.  The
// rows' bounds are read a lane each, a row's indices and values 32 at a time
// (coalesced, the next row's first ones ahead of time) and broadcast by
// shuffles, and the gathers of kSrpBatch nonzeros are issued together.  Rows of
// more than kSrpLongRow nonzeros are listed for srp_long_kernel: one of 7,700
// is a millisecond of one warp's time.
//
// Pieces: `outer` of them one after the other over all the rows, `inner` of
// them for a row at a time.  Where R exceeds L2 the columns are walked piece by
// piece (outer), so that a slice of R that fits L2 is gathered from at a time;
// otherwise all of a row's pieces follow each other (inner), which reads its
// indices once.
//
// The sum is formed in blocks of 32 nonzeros (a block's FMA chain, then the
// block added to the total), so a column's result carries at most min(n, 32) +
// ceil(n / 32) roundings in any chain rather than n.  Two-byte codes are summed
// as q - 2^15 in paired FP32 instructions, exactly decoded, in units of 2^-12;
// |q - 2^15| <= 2^15 bounds their magnitudes by 2^15 sum|v_i|, about ten times
// looser than each column's own sum, but rows are short here and it saves two
// paired FMAs and four masks a nonzero.  Float columns keep their own sums.
//
// What bounds it: the latency of the gathers of R's rows (one a nonzero, from
// L2 or HBM), so as many as the registers allow are in flight; with 64
// registers (four CTAs an SM) and eight gathers a batch the rows' kernel takes
// 4.37 ms on the 5e6 rows below, with 79 registers 6.46 ms, with four a batch
// 4.45 ms, with five CTAs 4.66 ms, and with the codes staged in shared memory
// by asynchronous copies 4.78 ms.
//
// 5e6 rows, 1.4e8 nonzeros, the first 256 columns of two-byte codes: 11.5 ms
// with four codes a lane and long rows left to single warps, now 4.41 ms + 3.36
// ms for the rows of more than 256 nonzeros and the rechecks (a kernel of their
// own before); 20,000 rows x 2,048 columns of floats (R of 820 MB) 607 us, now
// 518 us + 52 us; 7,000 rows x 128 codes 33 us a call, 44 with three launches.
constexpr int kSrpLongRow = 256;
constexpr int kSrpLongMost = 1024;

// The items' counters, 256 bytes apart in the context's scratch area.
constexpr unsigned kSrpCounters = 8;
__host__ __device__ __forceinline__ unsigned long long *srp_counter(blsh_dev_scratch *s, unsigned c) {
    return reinterpret_cast<unsigned long long *>(s->cta_counts) + 32 * c;
}

// Where a call's rows and columns lie, and its queues.
struct SrpArgs {
    const int64_t *indptr;
    const uint32_t *indices;
    const float *values;
    long long N, dim;
    int bits, col_first, outer, inner;
    int many;                  // (row, piece) items enough to fill the GPU several times
    const uint8_t *row_mask;   // rows to project (NULL: all)
    uint32_t *sig;
    blsh_dev_scratch *scratch;
    uint2 *queue;              // undecided signs, for srp_long_kernel
    unsigned long long *longs; // rows of more than kSrpLongRow nonzeros (BLSH_LITE_QUEUE_CAP of them)
};

// From how many nonzeros on a row is a CTA's: kSrpLongRow, but where there are
// rows for every warp anyway, four times the average row, up to kSrpLongMost.  A
// CTA's eight warps are half idle on a row of 300, and where most rows are as
// long that is most of the work (20,000 rows of 200 on average x 1,024 columns,
// R of 1,000 rows: 791 us with 256 for all, 677 here).
__device__ __forceinline__ int srp_long_row(const SrpArgs &A) {
    if (!A.many) return kSrpLongRow;
    const float four = 4.0f * (float)(__ldg(A.indptr + A.N) - __ldg(A.indptr)) / (float)A.N;
    return four > (float)kSrpLongMost ? kSrpLongMost : four > (float)kSrpLongRow ? (int)four : kSrpLongRow;
}

// A lane's CPL columns: their sums of a block, then of the row.
template <typename RT, int CPL>
struct SrpCols;
template <int CPL>
struct SrpCols<uint16_t, CPL> {
    static constexpr int W = CPL / 2;   // 32-bit words of codes
    unsigned long long acc[W], tot[W];
    uint32_t raw[kSrpBatch][W];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int i = 0; i < W; ++i) acc[i] = tot[i] = 0ull;
    }
    __device__ __forceinline__ void load(int b, const uint16_t *p) {
        if constexpr (W == 4) {
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(p));
            raw[b][0] = v.x; raw[b][1] = v.y; raw[b][2] = v.z; raw[b][3] = v.w;
        } else {
            const uint2 v = __ldg(reinterpret_cast<const uint2 *>(p));
            raw[b][0] = v.x; raw[b][1] = v.y;
        }
    }
    // the decoded value of code q is (q - 2^15) 2^-12: (2^23 + q) - (2^23 + 2^15), exact
    __device__ __forceinline__ void add(int b, float v) {
        const unsigned long long off2 = f2_pack(-8421376.0f, -8421376.0f), v2 = f2_pack(v, v);
#pragma unroll
        for (int i = 0; i < W; ++i) acc[i] = f2_fma(v2, f2_add(f2_codes(raw[b][i]), off2), acc[i]);
    }
    // with the magnitudes' sums in mag (pairs)
    __device__ __forceinline__ void add(int b, float v, unsigned long long (&mag)[W]) {
        const unsigned long long off2 = f2_pack(-8421376.0f, -8421376.0f), v2 = f2_pack(v, v);
        const unsigned long long av2 = f2_pack(fabsf(v), fabsf(v));
#pragma unroll
        for (int i = 0; i < W; ++i) {
            const unsigned long long d = f2_add(f2_codes(raw[b][i]), off2);
            acc[i] = f2_fma(v2, d, acc[i]);
            mag[i] = f2_fma(av2, d & 0x7fffffff7fffffffull, mag[i]);
        }
    }
    __device__ __forceinline__ void end_block() {
#pragma unroll
        for (int i = 0; i < W; ++i) {
            tot[i] = f2_add(tot[i], acc[i]);
            acc[i] = 0ull;
        }
    }
    __device__ __forceinline__ void totals(float (&t)[CPL]) const {
#pragma unroll
        for (int i = 0; i < W; ++i) f2_unpack(tot[i], t[2 * i], t[2 * i + 1]);
    }
};
template <int CPL>
struct SrpCols<float, CPL> {
    static_assert(CPL == 4, "16-byte loads of four columns");
    float acc[4], tot[4];
    float4 raw[kSrpBatch];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] = tot[i] = 0.0f;
    }
    __device__ __forceinline__ void load(int b, const float *p) { raw[b] = __ldg(reinterpret_cast<const float4 *>(p)); }
    __device__ __forceinline__ void add(int b, float v, float (&mag)[4]) {
        const float av = fabsf(v);
        const float r[4] = {raw[b].x, raw[b].y, raw[b].z, raw[b].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            acc[i] = __fmaf_rn(v, r[i], acc[i]);
            mag[i] = __fmaf_rn(av, fabsf(r[i]), mag[i]);
        }
    }
    __device__ __forceinline__ void end_block() {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            tot[i] = __fadd_rn(tot[i], acc[i]);
            acc[i] = 0.0f;
        }
    }
    __device__ __forceinline__ void totals(float (&t)[4]) const {
#pragma unroll
        for (int i = 0; i < 4; ++i) t[i] = tot[i];
    }
};

// The column sums' error bound: `chain` roundings in the longest chain (with
// its 25% slack good while n u <= 0.05), and up to 2n roundings near underflow.
__device__ __forceinline__ float srp_bound(float chain, float mag, float n) {
    return 1.25f * chain * 5.9604644775390625e-8f * mag + n * 1.4e-45f;
}

// An undecided sign: queued for srp_long_kernel (bit left 0), or summed in
// line if the queue is full.
template <typename RT>
__device__ __forceinline__ bool srp_undecided(const SrpArgs &A, const RT *R, long long row, long long s, long long e,
                                              int j, unsigned long long &rechecked, unsigned long long &zeros) {
    const unsigned long long slot = atomicAdd(&A.scratch->recheck_count, 1ull);
    if (slot < BLSH_RECHECK_CAP) {
        A.queue[slot] = make_uint2((uint32_t)row, (uint32_t)j);
        return false;
    }
    const double d = srp_recheck_fp64<RT>(A.indices, A.values, s, e, R, A.dim, A.bits, j);
    ++rechecked;
    zeros += d == 0.0;
    return d >= 0.0;
}

// GRABS 0: no more items than warps, a warp's is that of its number.  1: items
// from a counter.  8: counter c hands out items c, c + 8, ...  One counter takes
// about 0.9 ns a grab, the last and vain one of every warp included, which had
// been most of a masked call over 20,000 to 100,000 rows; rows that are all
// projected hide it (and the eight counters' addresses cost 3% there).
template <typename RT, int CPL, int GRABS>
__global__ void __launch_bounds__(256, 4) srp_sparse4_kernel(const SrpArgs A, const RT *__restrict__ R, int G) {
    constexpr bool Q16 = sizeof(RT) == 2;
    constexpr int PC = 32 * CPL;   // columns of a piece
    const int lane = threadIdx.x & 31;
    const int words = A.bits >> 5;
    unsigned long long rechecked = 0, zeros = 0, bad = 0;
    const int long_row = srp_long_row(A);
    const long long groups = (A.N + G - 1) / G;
    const unsigned long long items = (unsigned long long)groups * A.outer;
    for (;;) {
        unsigned long long item = 0;
        if constexpr (GRABS == 0) {
            item = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
        } else if constexpr (GRABS == 1) {
            if (lane == 0) item = atomicAdd(&A.scratch->hash_work, 1ull);
            item = __shfl_sync(kFull, item, 0);
        } else {
            if (lane == 0) item = GRABS * atomicAdd(srp_counter(A.scratch, blockIdx.x % GRABS), 1ull) + blockIdx.x % GRABS;
            item = __shfl_sync(kFull, item, 0);
        }
        if (item >= items) break;
        const int outer = A.outer == 1 ? 0 : (int)(item / (unsigned long long)groups);
        const long long r0 = ((long long)item - outer * groups) * G;
        // this grab's rows, a lane each
        long long my_s = 0;
        int my_len = 0;
        bool sel = false;
        if (lane < G && r0 + lane < A.N && (!A.row_mask || A.row_mask[r0 + lane])) {
            my_s = __ldg(A.indptr + r0 + lane);
            const long long len = __ldg(A.indptr + r0 + lane + 1) - my_s;
            sel = len <= long_row;
            my_len = sel ? (int)len : 0;
            if (!sel && outer == 0) {
                const unsigned long long slot = atomicAdd(&A.scratch->work3, 1ull);
                if (slot < BLSH_LITE_QUEUE_CAP) A.longs[slot] = (unsigned long long)(r0 + lane);
            }
        }
        unsigned todo = __ballot_sync(kFull, sel);
        uint32_t nx_ix = 0;
        float nx_v = 0.0f;
        auto first_block = [&](int l) {   // row l's first 32 nonzeros
            const long long s = __shfl_sync(kFull, my_s, l);
            const int len = __shfl_sync(kFull, my_len, l);
            nx_ix = 0;
            nx_v = 0.0f;
            if (lane < len) {
                nx_ix = __ldg(A.indices + s + lane);
                nx_v = __ldg(A.values + s + lane);
            }
        };
        if (todo) first_block(__ffs(todo) - 1);
        while (todo) {
            const int l = __ffs(todo) - 1;
            todo &= todo - 1;
            const long long row = r0 + l, s = __shfl_sync(kFull, my_s, l);
            const int len = __shfl_sync(kFull, my_len, l);
            uint32_t ix0 = nx_ix;
            float v0 = nx_v;
            if (todo) first_block(__ffs(todo) - 1);
            // malformed entries: counted once, contribute nothing
            auto check = [&](uint32_t &ix, float &v, bool count) {
                if (ix >= A.dim) {
                    bad += count;
                    ix = 0;
                    v = 0.0f;
                }
            };
            check(ix0, v0, outer == 0);
            for (int p = 0; p < A.inner; ++p) {
                const int col0 = A.col_first + (outer * A.inner + p) * PC;
                const RT *Rc = R + col0 + CPL * lane;
                SrpCols<RT, CPL> c;
                c.clear();
                [[maybe_unused]] float mag[CPL];
#pragma unroll
                for (int i = 0; i < CPL; ++i) mag[i] = 0.0f;
                float sav = 0.0f;   // this lane's part of sum|v|
                for (int k0 = 0; k0 < len; k0 += 32) {
                    uint32_t my_ix = ix0;
                    float my_v = v0;
                    if (k0) {
                        my_ix = 0;
                        my_v = 0.0f;
                        if (k0 + lane < len) {
                            my_ix = __ldg(A.indices + s + k0 + lane);
                            my_v = __ldg(A.values + s + k0 + lane);
                            check(my_ix, my_v, outer == 0 && p == 0);
                        }
                    }
                    if (Q16) sav += fabsf(my_v);
                    const int cnt = len - k0 < 32 ? len - k0 : 32;
                    for (int u0 = 0; u0 < cnt; u0 += kSrpBatch) {
                        float vb[kSrpBatch];
#pragma unroll
                        for (int b = 0; b < kSrpBatch; ++b) {   // (past the row's end: row 0 of R times 0)
                            const uint32_t ix = __shfl_sync(kFull, my_ix, (u0 + b) & 31);
                            vb[b] = __shfl_sync(kFull, my_v, (u0 + b) & 31);
                            c.load(b, Rc + (size_t)ix * A.bits);
                        }
#pragma unroll
                        for (int b = 0; b < kSrpBatch; ++b) {
                            if constexpr (Q16) c.add(b, vb[b]);
                            else c.add(b, vb[b], mag);
                        }
                    }
                    c.end_block();
                }
                float t[CPL];
                c.totals(t);
                if (Q16) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) sav += __shfl_xor_sync(kFull, sav, o);
                }
                const float n = (float)len;
                const float chain = fminf(n, 32.0f) + (float)((len + 31) >> 5);
                uint32_t word = 0;
#pragma unroll
                for (int i = 0; i < CPL; ++i) {
                    bool bit = t[i] >= 0.0f;
                    if (!(fabsf(t[i]) > srp_bound(chain, Q16 ? 32768.0f * sav : mag[i], n)))
                        bit = srp_undecided<RT>(A, R, row, s, s + len, col0 + CPL * lane + i, rechecked, zeros);
                    word |= (uint32_t)bit << i;
                }
                // 32 / CPL lanes' bits form a word
                word <<= CPL * (lane & (32 / CPL - 1));
#pragma unroll
                for (int o = 1; o < 32 / CPL; o <<= 1) word |= __shfl_xor_sync(kFull, word, o);
                if ((lane & (32 / CPL - 1)) == 0)
                    A.sig[(size_t)row * words + (col0 >> 5) + lane / (32 / CPL)] = word;
            }
        }
        if constexpr (GRABS == 0) break;
    }
    if (bad) blsh_dev_error(A.scratch, BLSH_ERANGE, 0, bad);
    if (rechecked) atomicAdd(&A.scratch->counters[2], rechecked);
    if (zeros) atomicAdd(&A.scratch->counters[3], zeros);
}

// An undecided sign, by the whole warp.  The lanes form the row's exact
// FP64 products (coalesced reads of the row, gathers of R) and sum them in
// parallel, together with their magnitudes: that sum errs by at most
// (n/32 + 5) u sum|p| (u = 2^-53), the oracle's row-order sum by at most
// (n - 1) u sum|p|, so a parallel sum larger than 1.25 (2n + 8) u sum|p| has
// the sign of the exact sum and of the oracle's.  Only the rest (exact zeros
// and ties within that bound) are summed in row order, one product at a
// time, which is the oracle's sum bit for bit.
template <typename RT>
__device__ __forceinline__ bool srp_sign_warp(const SrpArgs &A, const RT *__restrict__ R, long long s, long long e, int j,
                                              bool &zero) {
    const int lane = threadIdx.x & 31;
    // lane l sums entries l, l + 32, ... in that order, sixteen of its
    // gathers in flight at a time while more than 128 entries are left,
    // then four (a product of 0 for entries past the row leaves the sums
    // unchanged).  Four always: the longest rows' signs, 20,000 entries
    // each, held the kernel up (5e6 rows, 256 columns of codes: 375 us, 234
    // with sixteen; 20,000 rows of floats 20 and 14).
    double ps = 0.0, qs = 0.0;
    auto sum = [&](auto width, long long k0) {
        constexpr int U = decltype(width)::value;
        uint32_t ix[U];
        double p[U];
#pragma unroll
        for (int u = 0; u < U; ++u) ix[u] = k0 + 32 * u < e ? __ldg(A.indices + k0 + 32 * u) : 0xffffffffu;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            p[u] = 0.0;
            if (k0 + 32 * u < e && ix[u] < A.dim)
                p[u] = (double)__ldg(A.values + k0 + 32 * u) * r_fp64(R, (size_t)ix[u] * A.bits + j);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            ps += p[u];
            qs += fabs(p[u]);
        }
    };
    long long k0 = s + lane;
    for (; k0 - lane + 128 < e; k0 += 512) sum(std::integral_constant<int, 16>{}, k0);
    for (; k0 - lane < e; k0 += 128) sum(std::integral_constant<int, 4>{}, k0);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ps += __shfl_xor_sync(kFull, ps, o);
        qs += __shfl_xor_sync(kFull, qs, o);
    }
    const double len = (double)(e - s);
    zero = false;
    if (fabs(ps) > 1.25 * (2.0 * len + 8.0) * 1.1102230246251565e-16 * qs + (2.0 * len + 8.0) * 5e-324) return ps >= 0.0;
    // row order: lanes load 32 products at a time, every lane adds them in order
    double d = 0.0;
    for (long long c0 = s; c0 < e; c0 += 32) {
        double p = 0.0;
        if (c0 + lane < e) {
            const uint32_t ix = __ldg(A.indices + c0 + lane);
            if (ix < A.dim) p = (double)__ldg(A.values + c0 + lane) * r_fp64(R, (size_t)ix * A.bits + j);
        }
        const int cnt = (int)min(32ll, e - c0);
        for (int l = 0; l < cnt; ++l) d += __shfl_sync(kFull, p, l);
    }
    zero = d == 0.0;
    return d >= 0.0;
}

// Rows of more than kSrpLongRow nonzeros: a CTA per (row, piece), handed out
// from a counter, its eight warps taking every eighth block of 32 nonzeros; the
// warps' sums and magnitudes (every column's own here) meet in shared memory,
// added in warp order.  No product passes through more than 32 + ceil(n / 256)
// + 8 roundings.  A warp's undecided columns are decided at once, and when the
// long rows have been handed out the signs that the rows' kernel queued (a
// warp each; a nonnegative sum sets the bit, the word was written with it
// clear): a launch of their own cost a small call 7 to 10 us.
template <typename RT, int CPL>
__global__ void __launch_bounds__(256, 3) srp_long_kernel(const SrpArgs A, const RT *__restrict__ R) {
    constexpr int PC = 32 * CPL;
    __shared__ float s_tot[8][PC], s_mag[8][PC];
    __shared__ unsigned long long s_item;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int words = A.bits >> 5, pieces = A.outer * A.inner;
    const unsigned long long listed = A.scratch->work3;
    const bool all = listed > BLSH_LITE_QUEUE_CAP;   // more than the list holds: every row is looked at
    const unsigned long long items = (all ? (unsigned long long)A.N : listed) * pieces;
    unsigned long long rechecked = 0, zeros = 0, bad = 0;
    while (items > 0) {                               // (no grab where no row is long)
        __syncthreads();                              // the previous item and its sums have been read
        if (threadIdx.x == 0) s_item = atomicAdd(&A.scratch->work2, 1ull);
        __syncthreads();
        const unsigned long long item = s_item;
        if (item >= items) break;
        const unsigned long long q = item / (unsigned)pieces;
        const int p = (int)(item - q * (unsigned)pieces);
        const long long row = (long long)(all ? q : A.longs[q]);
        if (all && A.row_mask && !A.row_mask[row]) continue;
        const long long s = __ldg(A.indptr + row), len = __ldg(A.indptr + row + 1) - s;
        if (all && len <= srp_long_row(A)) continue;   // (a listed row is long)
        const int col0 = A.col_first + p * PC;
        const RT *Rc = R + col0 + CPL * lane;
        SrpCols<RT, CPL> c;
        c.clear();
        float mag[CPL];
#pragma unroll
        for (int i = 0; i < CPL; ++i) mag[i] = 0.0f;
        [[maybe_unused]] unsigned long long mag2[CPL / 2];
#pragma unroll
        for (int i = 0; i < CPL / 2; ++i) mag2[i] = 0ull;
        for (long long k0 = 32 * warp; k0 < len; k0 += 256) {
            uint32_t my_ix = 0;
            float my_v = 0.0f;
            if (k0 + lane < len) {
                my_ix = __ldg(A.indices + s + k0 + lane);
                my_v = __ldg(A.values + s + k0 + lane);
                if (my_ix >= A.dim) {
                    bad += p == 0;
                    my_ix = 0;
                    my_v = 0.0f;
                }
            }
            const int cnt = len - k0 < 32 ? (int)(len - k0) : 32;
            for (int u0 = 0; u0 < cnt; u0 += kSrpBatch) {
                float vb[kSrpBatch];
#pragma unroll
                for (int b = 0; b < kSrpBatch; ++b) {
                    const uint32_t ix = __shfl_sync(kFull, my_ix, (u0 + b) & 31);
                    vb[b] = __shfl_sync(kFull, my_v, (u0 + b) & 31);
                    c.load(b, Rc + (size_t)ix * A.bits);
                }
#pragma unroll
                for (int b = 0; b < kSrpBatch; ++b) {
                    if constexpr (sizeof(RT) == 2) c.add(b, vb[b], mag2);
                    else c.add(b, vb[b], mag);
                }
            }
            c.end_block();
        }
        float t[CPL];
        c.totals(t);
        if constexpr (sizeof(RT) == 2) {
#pragma unroll
            for (int i = 0; i < CPL / 2; ++i) f2_unpack(mag2[i], mag[2 * i], mag[2 * i + 1]);
        }
#pragma unroll
        for (int i = 0; i < CPL; ++i) {
            s_tot[warp][CPL * lane + i] = t[i];
            s_mag[warp][CPL * lane + i] = mag[i];
        }
        __syncthreads();
        if (threadIdx.x < PC) {
            float tt = 0.0f, mm = 0.0f;
#pragma unroll
            for (int w = 0; w < 8; ++w) {
                tt = __fadd_rn(tt, s_tot[w][threadIdx.x]);
                mm = __fadd_rn(mm, s_mag[w][threadIdx.x]);
            }
            // the row length through a 32-bit integer; rows past 2^30 count as 2^30, which is too long
            const int len32 = (int)(len < (1ll << 30) ? len : (1ll << 30));
            const float n = (float)len32;
            const bool too_long = n * 5.9604644775390625e-8f > 0.05f;   // the 1.25 slack needs n u <= 0.05
            const float chain = 40.0f + (float)((len32 + 255) >> 8);
            unsigned word = __ballot_sync(kFull, tt >= 0.0f);
            for (unsigned open = __ballot_sync(kFull, too_long || !(fabsf(tt) > srp_bound(chain, mm, n))); open;
                 open &= open - 1) {
                const int c = __ffs(open) - 1;
                bool zero;
                const bool bit = srp_sign_warp<RT>(A, R, s, s + len, col0 + 32 * warp + c, zero);
                word = bit ? word | 1u << c : word & ~(1u << c);
                rechecked += lane == 0;
                zeros += lane == 0 && zero;
            }
            if (lane == 0) A.sig[(size_t)row * words + (col0 >> 5) + warp] = word;
        }
    }
    // the queued signs
    const unsigned long long total = A.scratch->recheck_count;
    const unsigned long long n = total < BLSH_RECHECK_CAP ? total : BLSH_RECHECK_CAP;
    const unsigned long long warps = (unsigned long long)gridDim.x * (blockDim.x >> 5);
    for (unsigned long long it = (unsigned long long)blockIdx.x * (blockDim.x >> 5) + warp; it < n; it += warps) {
        const uint2 rj = A.queue[it];
        bool zero;
        const bool bit = srp_sign_warp<RT>(A, R, __ldg(A.indptr + rj.x), __ldg(A.indptr + rj.x + 1), (int)rj.y, zero);
        if (lane == 0) {
            if (bit) atomicOr(A.sig + (size_t)rj.x * words + (rj.y >> 5), 1u << (rj.y & 31));
            ++rechecked;
            zeros += zero;
        }
    }
    if (bad) blsh_dev_error(A.scratch, BLSH_ERANGE, 0, bad);
    if (rechecked) atomicAdd(&A.scratch->counters[2], rechecked);
    if (zeros) atomicAdd(&A.scratch->counters[3], zeros);
}

// Two-byte codes of Gaussian samples (Section 4.3): q = floor((x + 8) 2^12),
// formed as floor(x 2^12) + 2^15 (exact in FP32).  Codes outside [0, 65535]
// (x < -8 or x >= 8) and NaN are clamped (NaN to 0) and reported.
__global__ void __launch_bounds__(256) quantize_gaussian_kernel(const float *__restrict__ x, long long n,
                                                                uint16_t *__restrict__ q, blsh_dev_scratch *scratch) {
    unsigned long long outside = 0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        float c = floorf(__ldg(x + i) * 4096.0f) + 32768.0f;
        if (!(c >= 0.0f)) {
            c = 0.0f;
            ++outside;
        } else if (c > 65535.0f) {
            c = 65535.0f;
            ++outside;
        }
        q[i] = (uint16_t)c;
    }
    if (outside) blsh_dev_error(scratch, BLSH_ENUMERIC, -1, outside);
}

// SplitMix64 (Steele, Lea and Flood 2014) read as a counter-based
// generator: output k of the stream `seed` is the finaliser of
// seed + (k + 1) * 0x9E3779B97F4A7C15.
__device__ __forceinline__ unsigned long long splitmix64_at(unsigned long long seed, unsigned long long k) {
    unsigned long long z = seed + (k + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Eight codes per thread (one 16-byte store): entry c = t * bits + j sums
// the twelve 16-bit pieces of outputs 3c .. 3c+2 (Irwin-Hall, mean 393210,
// standard deviation 65536 to 1e-10) and encodes x = (S - 393210) / 2^16 as
// floor((x + 8) 2^16 / 16) = floor((S - 393210) / 16) + 32768.
__global__ void __launch_bounds__(256) gaussian_codes_kernel(unsigned long long seed, long long groups,
                                                             uint16_t *__restrict__ codes) {
    for (long long gidx = (long long)blockIdx.x * blockDim.x + threadIdx.x; gidx < groups;
         gidx += (long long)gridDim.x * blockDim.x) {
        uint32_t packed[4];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const unsigned long long c = (unsigned long long)gidx * 8ull + (unsigned long long)e;
            int S = 0;
#pragma unroll
            for (int w = 0; w < 3; ++w) {
                const unsigned long long o = splitmix64_at(seed, 3ull * c + (unsigned long long)w);
                S += (int)(o & 0xFFFFull) + (int)((o >> 16) & 0xFFFFull) + (int)((o >> 32) & 0xFFFFull) +
                     (int)(o >> 48);
            }
            const int code = ((S - 393210) >> 4) + 32768;   // arithmetic shift: floor division by 16
            if (e & 1) packed[e >> 1] |= (uint32_t)code << 16;
            else packed[e >> 1] = (uint32_t)code;
        }
        reinterpret_cast<uint4 *>(codes)[gidx] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
    }
}

// Dense rows X [N][d] against R [d][bits] on the CUDA cores: the shapes the
// tensor-core path does not take (bits no multiple of 256, no workspace,
// unaligned rows).  A CTA of 256 threads forms a tile of 8 RT rows by 128
// columns, K in stages of 32 staged in shared memory (X turned, so that a
// thread reads its RT rows' values of a coordinate in 16-byte loads that the
// whole warp shares); thread t owns rows RT (t / 32) .. and columns
// 4 (t % 32) .. +3.  With RT = 8 a coordinate costs a thread 32 FMAs for
// three 16-byte shared loads, and R is read from L2 once per 64 rows; the
// former kernel (one row per CTA, R streamed from L2 for every row, a second
// FMA per product for the error bound) was bound by those reads: 99,991 x 300
// x 1,024 bits took 36.4 ms, 2.61 ms here; 1,659 x 100 x 512 bits 208 us, 29 us here.
//
// Error bound: a stage's chain of at most 32 FMAs, then the stage totals
// added in order, so no product passes through more than 32 + ceil(d/32)
// roundings, and sum|x_i r_ij| <= |x| |r_j| (norms formed from the staged
// values, every operation rounded up): a sum of magnitude above 1.25 times
// that many u |x| |r_j| (plus the underflow terms) has the sign of the exact
// sum.  The others, about 1 in 10^4, are listed and summed in FP64 over
// coordinates 0..d-1 in order, which is the definition, a thread each: where a
// tenth of the sums are ties (rows of +-1, 100 x 64 x 128 bits) a lane summing
// its own took 223 us, 35 so.  Zero rows and columns need no sum.
constexpr int kSimtK = 32;
constexpr int kSimtCols = 128;

template <int RT>
__global__ void __launch_bounds__(256) srp_dense_simt_kernel(const float *__restrict__ X, long long N, int d,
                                                             const float *__restrict__ R, int bits, int col_tiles,
                                                             uint32_t *__restrict__ sig, blsh_dev_scratch *scratch) {
    constexpr int ROWS = 8 * RT;
    __shared__ __align__(16) float xs[kSimtK][ROWS + 4];      // [k][row]
    __shared__ __align__(16) float rs[kSimtK][kSimtCols];
    __shared__ float xn[ROWS], rn[kSimtCols];
    __shared__ int s_open;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const long long rt = blockIdx.x / col_tiles;
    const int j0 = (int)(blockIdx.x - rt * col_tiles) * kSimtCols;
    const long long row0 = rt * ROWS;
    const int ncols = bits - j0 < kSimtCols ? bits - j0 : kSimtCols;   // a multiple of 32
    float tot[RT][4];
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) tot[i][c] = 0.0f;
    float nrm = 0.0f;   // threads 0 .. ROWS-1: their row's squared norm; 128 .. 255: their column's
    if (t == 0) s_open = 0;
    for (int k0 = 0; k0 < d; k0 += kSimtK) {
        const int kn = d - k0 < kSimtK ? (d - k0 + 7) & ~7 : kSimtK;   // (whole eights: the loops below)
        __syncthreads();
        if (lane < kn)
            for (int r = w; r < ROWS; r += 8) {
                const long long row = row0 + r;
                xs[lane][r] = row < N && k0 + lane < d ? __ldg(X + (size_t)row * d + k0 + lane) : 0.0f;
            }
        for (int i = t; i < kn * kSimtCols; i += 256) {
            const int k = i / kSimtCols, c = i % kSimtCols;
            rs[k][c] = k0 + k < d && c < ncols ? __ldg(R + (size_t)(k0 + k) * bits + j0 + c) : 0.0f;
        }
        __syncthreads();
        if (t < ROWS) {
            for (int k8 = 0; k8 < kn; k8 += 8)
#pragma unroll
                for (int k = k8; k < k8 + 8; ++k) nrm = __fmaf_ru(xs[k][t], xs[k][t], nrm);
        } else if (t >= 128) {
            for (int k8 = 0; k8 < kn; k8 += 8)
#pragma unroll
                for (int k = k8; k < k8 + 8; ++k) nrm = __fmaf_ru(rs[k][t - 128], rs[k][t - 128], nrm);
        }
        float acc[RT][4];
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[i][c] = 0.0f;
        for (int k8 = 0; k8 < kn; k8 += 8)
#pragma unroll
            for (int k = k8; k < k8 + 8; ++k) {
                const float4 r = *reinterpret_cast<const float4 *>(&rs[k][4 * lane]);
                float x[RT];
#pragma unroll
                for (int i = 0; i < RT; i += 4) {
                    const float4 v = *reinterpret_cast<const float4 *>(&xs[k][RT * w + i]);
                    x[i] = v.x; x[i + 1] = v.y; x[i + 2] = v.z; x[i + 3] = v.w;
                }
#pragma unroll
                for (int i = 0; i < RT; ++i) {
                    acc[i][0] = __fmaf_rn(x[i], r.x, acc[i][0]);
                    acc[i][1] = __fmaf_rn(x[i], r.y, acc[i][1]);
                    acc[i][2] = __fmaf_rn(x[i], r.z, acc[i][2]);
                    acc[i][3] = __fmaf_rn(x[i], r.w, acc[i][3]);
                }
            }
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int c = 0; c < 4; ++c) tot[i][c] = __fadd_rn(tot[i][c], acc[i][c]);
    }
    if (t < ROWS) xn[t] = __fsqrt_ru(nrm);
    else if (t >= 128) rn[t - 128] = __fsqrt_ru(nrm);
    __syncthreads();
    const int words = bits >> 5;
    const float u = 1.25f * (float)(kSimtK + (d + kSimtK - 1) / kSimtK) * 5.9604644775390625e-8f;
    const float tiny = (float)d * 2.9e-45f;
    const bool loose = (float)d * 5.9604644775390625e-8f > 0.05f;   // the 1.25 slack needs d u <= 0.05
    // the decided bits into shared memory, the open signs (row of the tile << 7 |
    // column) into a list there: one sum a thread, so that rows of ties are not
    // one lane's sixteen or thirty-two sums one after the other
    auto s_bits = reinterpret_cast<uint32_t(*)[kSimtCols / 32]>(&xs[0][0]);   // [ROWS][4]
    uint16_t *s_list = reinterpret_cast<uint16_t *>(&rs[0][0]);               // [ROWS * 128]
    static_assert(ROWS * kSimtCols * sizeof(uint16_t) <= sizeof(rs) && ROWS * 16 <= sizeof(xs), "the stage's place");
    uint32_t open = 0;   // bit 4 i + c
    unsigned long long rechecked = 0, zeros = 0;
#pragma unroll
    for (int i = 0; i < RT; ++i) {
        const long long row = row0 + RT * w + i;
        const float xi = xn[RT * w + i], ux = u * xi;
        uint32_t nib = 0;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int col = 4 * lane + c;
            const bool decided = !loose && fabsf(tot[i][c]) > ux * rn[col] + tiny;
            // (zeros against finite values: every product is zero; no square is lost in the norms)
            const bool zero = xi * rn[col] == 0.0f && (xi == 0.0f || rn[col] == 0.0f);
            if (row < N && col < ncols && !decided) {
                if (zero) ++zeros;
                else open |= 1u << (4 * i + c);
            }
            nib |= (uint32_t)(zero || (decided && tot[i][c] >= 0.0f)) << c;
        }
        // eight lanes' nibbles form a word
        uint32_t word = nib << (4 * (lane & 7));
        word |= __shfl_xor_sync(kFull, word, 1);
        word |= __shfl_xor_sync(kFull, word, 2);
        word |= __shfl_xor_sync(kFull, word, 4);
        if ((lane & 7) == 0) s_bits[RT * w + i][lane >> 3] = word;
    }
    const int mine = __popc(open);
    int before = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, before, o);
        if (lane >= o) before += y;
    }
    int at = 0;
    if (lane == 31 && before) at = atomicAdd(&s_open, before);
    at = __shfl_sync(kFull, at, 31) + before - mine;
    for (; open; open &= open - 1) {
        const int b = __ffs(open) - 1;
        s_list[at++] = (uint16_t)((RT * w + (b >> 2)) << 7 | (4 * lane + (b & 3)));
    }
    __syncthreads();
    rechecked = zeros;
    for (int e = t; e < s_open; e += 256) {
        const int r = s_list[e] >> 7, col = s_list[e] & 127;
        const float *x = X + (size_t)(row0 + r) * d, *rc = R + j0 + col;
        double dd = 0.0;
#pragma unroll 4
        for (int k = 0; k < d; ++k) dd += (double)__ldg(x + k) * (double)__ldg(rc + (size_t)k * bits);
        if (dd >= 0.0) atomicOr(&s_bits[r][col >> 5], 1u << (col & 31));
        ++rechecked;
        zeros += dd == 0.0;
    }
    __syncthreads();
    for (int i = t; i < ROWS * (kSimtCols / 32); i += 256) {
        const int r = i >> 2, q = i & 3;
        if (row0 + r < N && 32 * q < ncols) sig[(size_t)(row0 + r) * words + (j0 >> 5) + q] = s_bits[r][q];
    }
    if (rechecked) atomicAdd(&scratch->counters[2], rechecked);
    if (zeros) atomicAdd(&scratch->counters[3], zeros);
}

// Columns [col0, col0 + ncols) of the sparse projection (multiples of 128) for
// the rows row_mask selects, on the aligned path.
template <typename RT, int CPL>
int srp_sparse_pieces(blsh_ctx *ctx, const int64_t *indptr, const uint32_t *indices, const float *values, int64_t N,
                      const RT *R, int64_t dim, int bits, int col0, int ncols, const uint8_t *row_mask,
                      uint32_t *sig, cudaStream_t s) {
    const int pieces = ncols / (32 * CPL);
    const long long warps = (long long)ctx->sm_count * 32;   // about the resident ones
    SrpArgs A;
    A.indptr = indptr;
    A.indices = indices;
    A.values = values;
    A.N = N;
    A.dim = dim;
    A.bits = bits;
    A.col_first = col0;
    A.row_mask = row_mask;
    A.sig = sig;
    A.scratch = ctx->scratch;
    A.queue = ctx->recheck_queue;
    A.longs = ctx->lite_queue;
    // piece by piece over all the rows where R's columns exceed half of L2, or
    // where there are too few rows to give every warp several
    const bool by_piece = (!row_mask && (double)dim * ncols * sizeof(RT) > 64e6) || N < 8 * warps;
    A.outer = by_piece ? pieces : 1;
    A.inner = by_piece ? 1 : pieces;
    A.many = N * pieces >= 4 * warps && !row_mask;
    // rows a grab: up to 32, about eight grabs a warp, four where a mask may leave
    // them next to nothing
    const long long grabs = (row_mask ? 4 : 8) * warps;
    int G = 32;
    while (G > 1 && (N / G) * A.outer < grabs) G >>= 1;
    blsh_dev_scratch *scr = ctx->scratch;
    // work2 (next long row), work3 (long rows listed), recheck_count .. the items' counters
    BLSH_CUDA(ctx, cudaMemsetAsync(&scr->work2, 0, (char *)(srp_counter(scr, kSrpCounters - 1) + 1) - (char *)&scr->work2, s));
    const char *name = sizeof(RT) == 2 ? "srp_sparse4_kernel (two-byte codes)" : "srp_sparse4_kernel";
    const long long items = (N + G - 1) / G * A.outer, blocks = (items + 7) / 8, most = (long long)ctx->sm_count * 8;
    blsh_time_start(ctx, s);
    const unsigned grid = (unsigned)(blocks < most ? blocks : most);
    if (items <= warps) srp_sparse4_kernel<RT, CPL, 0><<<grid, 256, 0, s>>>(A, R, G);
    else if (!row_mask) srp_sparse4_kernel<RT, CPL, 1><<<grid, 256, 0, s>>>(A, R, G);
    else srp_sparse4_kernel<RT, CPL, (int)kSrpCounters><<<grid, 256, 0, s>>>(A, R, G);
    BLSH_LAUNCHED(ctx, name);
    blsh_time_start(ctx, s);
    srp_long_kernel<RT, CPL><<<ctx->sm_count * 3, 256, 0, s>>>(A, R);
    BLSH_LAUNCHED(ctx, name);
    return BLSH_OK;
}

int srp_sparse_cols(blsh_ctx *ctx, const int64_t *indptr, const uint32_t *indices, const float *values, int64_t N,
                    const float *R, int64_t dim, int bits, int col0, int ncols, const uint8_t *row_mask,
                    uint32_t *sig, cudaStream_t s) {
    return srp_sparse_pieces<float, 4>(ctx, indptr, indices, values, N, R, dim, bits, col0, ncols, row_mask, sig, s);
}
int srp_sparse_cols(blsh_ctx *ctx, const int64_t *indptr, const uint32_t *indices, const float *values, int64_t N,
                    const uint16_t *R, int64_t dim, int bits, int col0, int ncols, const uint8_t *row_mask,
                    uint32_t *sig, cudaStream_t s) {
    // eight codes a lane where the pieces and the alignment allow it
    if (ncols % 256 == 0 && blsh_aligned(R, 16))
        return srp_sparse_pieces<uint16_t, 8>(ctx, indptr, indices, values, N, R, dim, bits, col0, ncols, row_mask, sig,
                                              s);
    return srp_sparse_pieces<uint16_t, 4>(ctx, indptr, indices, values, N, R, dim, bits, col0, ncols, row_mask, sig, s);
}

int srp_threads(int bits, int *per_thread) {
    const int words = bits / 32;
    int wt = 8;
    while (words % wt) --wt;
    *per_thread = bits / (32 * wt);
    return 32 * wt;
}

}  // namespace

// minhash_kernel over every set, then minhash_big_kernel over the long sets
// the first one listed.
template <int HPL>
int minhash_launch(blsh_ctx *ctx, cudaStream_t s, const int64_t *indptr, const uint32_t *indices, int64_t N,
                   int n_hashes, const uint32_t *a, const uint32_t *b, uint32_t *sig, const LongSets &L) {
    const unsigned tiles = (unsigned)(n_hashes / (32 * HPL));
    const long long blocks = (N + 7) / 8, cap = (long long)ctx->sm_count * 32;
    blsh_time_start(ctx, s);
    // a CTA per set where a warp per set would give an SM fewer than 32: then
    // the longest set's chain decides (2,000 sets, mean 50, longest 837, x 256
    // hashes: 124 us with a warp per set, 23 us with a CTA)
    if (N * tiles < 32ll * ctx->sm_count)
        minhash_cta_kernel<HPL><<<dim3((unsigned)N, tiles), 256, 0, s>>>(indptr, indices, n_hashes, a, b, sig, L);
    else
        minhash_kernel<HPL><<<dim3((unsigned)(blocks < cap ? blocks : cap), tiles < 65535u ? tiles : 65535u), 256, 0, s>>>(
            indptr, indices, N, n_hashes, a, b, sig, L);
    BLSH_LAUNCHED(ctx, "minhash_kernel");
    blsh_time_start(ctx, s);
    minhash_big_kernel<HPL><<<ctx->sm_count * 4, 256, 0, s>>>(indptr, indices, N, n_hashes, a, b, sig, L);
    BLSH_LAUNCHED(ctx, "minhash_big_kernel");
    return BLSH_OK;
}

extern "C" int blsh_minhash(blsh_ctx *ctx, const int64_t *indptr, const uint32_t *indices, int64_t N,
                            int32_t n_hashes, const uint32_t *a, const uint32_t *b, uint32_t *sig, void *stream) {
    if (!ctx) return BLSH_EINVAL;
    if (!indptr || !indices || !a || !b || !sig)
        return blsh_fail(ctx, BLSH_EINVAL, "indptr, indices, a, b and sig are required");
    if (N < 0 || n_hashes <= 0 || n_hashes % 32)
        return blsh_fail(ctx, BLSH_EINVAL, "n_hashes must be a positive multiple of 32");
    if (!blsh_aligned(indptr, 8)) return blsh_fail(ctx, BLSH_EINVAL, "misaligned indptr");
    if (N == 0) return BLSH_OK;
    blsh_device_guard g(ctx->device);
    cudaStream_t s = blsh_stream(stream);
    const int words = n_hashes / 32;
    // long sets go to minhash_big_kernel through the context's queues
    blsh_dev_scratch *scr = ctx->scratch;
    static_assert(offsetof(blsh_dev_scratch, work2) == offsetof(blsh_dev_scratch, work) + 8 &&
                      offsetof(blsh_dev_scratch, work3) == offsetof(blsh_dev_scratch, work) + 16 &&
                      offsetof(blsh_dev_scratch, recheck_count) == offsetof(blsh_dev_scratch, work) + 24,
                  "cleared together");
    const LongSets L = {reinterpret_cast<uint2 *>(ctx->lite_queue), ctx->recheck_queue, &scr->work3, &scr->recheck_count,
                        &scr->work};
    BLSH_CUDA(ctx, cudaMemsetAsync(&scr->work, 0, 4 * sizeof(unsigned long long), s));
    const int hpl = words % 8 == 0 ? 8 : words % 4 == 0 ? 4 : words % 2 == 0 ? 2 : 1;   // hashes a lane
    switch (hpl) {
    case 8: return minhash_launch<8>(ctx, s, indptr, indices, N, n_hashes, a, b, sig, L);
    case 4: return minhash_launch<4>(ctx, s, indptr, indices, N, n_hashes, a, b, sig, L);
    case 2: return minhash_launch<2>(ctx, s, indptr, indices, N, n_hashes, a, b, sig, L);
    default: return minhash_launch<1>(ctx, s, indptr, indices, N, n_hashes, a, b, sig, L);
    }
}

extern "C" int blsh_srp_sparse(blsh_ctx *ctx, const int64_t *indptr, const uint32_t *indices, const float *values,
                               int64_t N, const float *R, int64_t dim, int32_t bits, uint32_t *sig, void *stream) {
    if (!ctx) return BLSH_EINVAL;
    if (!indptr || !indices || !values || !R || !sig)
        return blsh_fail(ctx, BLSH_EINVAL, "indptr, indices, values, R and sig are required");
    if (N < 0 || N >= (1ll << 32) || dim <= 0 || bits <= 0 || bits % 32 || bits > 4096)
        return blsh_fail(ctx, BLSH_EINVAL, "bits must be a positive multiple of 32, at most 4096; N < 2^32");
    if (!blsh_aligned(indptr, 8)) return blsh_fail(ctx, BLSH_EINVAL, "misaligned indptr");
    if (N == 0) return BLSH_OK;
    // threads = 32 * (largest divisor of bits/32 that is at most 8)
    const int words = bits / 32;
    int wt = 8;
    while (words % wt) --wt;
    const int T = 32 * wt;
    const int per_thread = bits / T;
    if (per_thread > kSrpMaxPerThread) return blsh_fail(ctx, BLSH_EINVAL, "bits/32 needs a divisor in 2..8");
    blsh_device_guard g(ctx->device);
    cudaStream_t s = blsh_stream(stream);
    // many small CTAs (rows have very different lengths): 32 per SM measured best
    const long long cap = (long long)ctx->sm_count * 32;
    const unsigned grid = (unsigned)(N < cap ? N : cap);
    if (bits % 128 == 0 && blsh_aligned(R, 16))
        return srp_sparse_cols(ctx, indptr, indices, values, N, R, dim, bits, 0, bits, nullptr, sig, s);
    blsh_time_start(ctx, s);
    srp_sparse_kernel<float><<<grid, T, 0, s>>>(indptr, indices, values, N, R, dim, bits, per_thread, sig, ctx->scratch);
    BLSH_LAUNCHED(ctx, "srp_sparse_kernel");
    return BLSH_OK;
}

int blsh_srp_dense_simt(blsh_ctx *ctx, const float *X, int64_t N, int32_t d, const float *R, int32_t bits,
                        uint32_t *sig, cudaStream_t s) {
    int per_thread = 0;
    srp_threads(bits, &per_thread);
    // (the tiles could form either; the refusals are the entry point's: the sparse
    // projections take no such width, and rows have always been limited to 58,112 coordinates)
    if (per_thread > kSrpMaxPerThread) return blsh_fail(ctx, BLSH_EINVAL, "bits/32 needs a divisor in 2..8");
    if (sizeof(float) * (size_t)d > ctx->smem_optin) return blsh_fail(ctx, BLSH_EINVAL, "d too large");
    // 64-row tiles where they give every SM at least two, else 32-row ones
    const int col_tiles = (bits + kSimtCols - 1) / kSimtCols;
    const bool wide = (N + 63) / 64 * col_tiles >= 2ll * ctx->sm_count;
    const long long tiles = (wide ? (N + 63) / 64 : (N + 31) / 32) * col_tiles;   // N < 2^32, so < 2^31
    blsh_time_start(ctx, s);
    (wide ? srp_dense_simt_kernel<8> : srp_dense_simt_kernel<4>)<<<(unsigned)tiles, 256, 0, s>>>(
        X, N, d, R, bits, col_tiles, sig, ctx->scratch);
    BLSH_LAUNCHED(ctx, "srp_dense_simt_kernel");
    return BLSH_OK;
}

extern "C" int blsh_quantize_gaussian(blsh_ctx *ctx, const float *x, int64_t n, uint16_t *q, void *stream) {
    if (!ctx) return BLSH_EINVAL;
    if (n < 0 || (n > 0 && (!x || !q))) return blsh_fail(ctx, BLSH_EINVAL, "x and q are required");
    if (n == 0) return BLSH_OK;
    blsh_device_guard g(ctx->device);
    cudaStream_t s = blsh_stream(stream);
    const long long blocks = (n + 255) / 256;
    const long long cap = (long long)ctx->sm_count * 16;
    blsh_time_start(ctx, s);
    quantize_gaussian_kernel<<<(unsigned)(blocks < cap ? blocks : cap), 256, 0, s>>>(x, n, q, ctx->scratch);
    BLSH_LAUNCHED(ctx, "quantize_gaussian_kernel");
    return BLSH_OK;
}

extern "C" int blsh_gaussian_codes(blsh_ctx *ctx, uint64_t seed, int64_t dim, int32_t bits, uint16_t *codes,
                                   void *stream) {
    if (!ctx) return BLSH_EINVAL;
    if (dim < 0 || bits <= 0 || bits % 8 || (dim > 0 && !codes))
        return blsh_fail(ctx, BLSH_EINVAL, "bits must be a positive multiple of 8; codes are required");
    if (!blsh_aligned(codes, 16)) return blsh_fail(ctx, BLSH_EINVAL, "codes must be 16-byte aligned");
    if (dim == 0) return BLSH_OK;
    blsh_device_guard g(ctx->device);
    cudaStream_t s = blsh_stream(stream);
    const long long groups = dim * (long long)(bits / 8);
    const long long blocks = (groups + 255) / 256;
    const long long cap = (long long)ctx->sm_count * 32;
    blsh_time_start(ctx, s);
    gaussian_codes_kernel<<<(unsigned)(blocks < cap ? blocks : cap), 256, 0, s>>>((unsigned long long)seed, groups,
                                                                                  codes);
    BLSH_LAUNCHED(ctx, "gaussian_codes_kernel");
    return BLSH_OK;
}

extern "C" int blsh_srp_sparse_cols(blsh_ctx *ctx, const int64_t *indptr, const uint32_t *indices,
                                    const float *values, int64_t N, const float *R, int64_t dim, int32_t bits,
                                    int32_t col_begin, int32_t col_count, const uint8_t *row_mask, uint32_t *sig,
                                    void *stream) {
    if (!ctx) return BLSH_EINVAL;
    if (!indptr || !indices || !values || !R || !sig)
        return blsh_fail(ctx, BLSH_EINVAL, "indptr, indices, values, R and sig are required");
    if (N < 0 || N >= (1ll << 32) || dim <= 0 || bits <= 0 || bits % 128 || bits > 4096 || col_begin < 0 ||
        col_count <= 0 || col_begin % 128 || col_count % 128 || col_begin + col_count > bits)
        return blsh_fail(ctx, BLSH_EINVAL, "bits, col_begin and col_count must be multiples of 128 within bits");
    if (!blsh_aligned(indptr, 8) || !blsh_aligned(R, 16)) return blsh_fail(ctx, BLSH_EINVAL, "misaligned pointer");
    if (N == 0) return BLSH_OK;
    blsh_device_guard g(ctx->device);
    return srp_sparse_cols(ctx, indptr, indices, values, N, R, dim, bits, col_begin, col_count, row_mask,
                                   sig, blsh_stream(stream));
}

extern "C" int blsh_srp_sparse_q16_cols(blsh_ctx *ctx, const int64_t *indptr, const uint32_t *indices,
                                        const float *values, int64_t N, const uint16_t *Rq, int64_t dim,
                                        int32_t bits, int32_t col_begin, int32_t col_count,
                                        const uint8_t *row_mask, uint32_t *sig, void *stream) {
    if (!ctx) return BLSH_EINVAL;
    if (!indptr || !indices || !values || !Rq || !sig)
        return blsh_fail(ctx, BLSH_EINVAL, "indptr, indices, values, Rq and sig are required");
    if (N < 0 || N >= (1ll << 32) || dim <= 0 || bits <= 0 || bits % 128 || bits > 4096 || col_begin < 0 ||
        col_count <= 0 || col_begin % 128 || col_count % 128 || col_begin + col_count > bits)
        return blsh_fail(ctx, BLSH_EINVAL, "bits, col_begin and col_count must be multiples of 128 within bits");
    if (!blsh_aligned(indptr, 8) || !blsh_aligned(Rq, 8)) return blsh_fail(ctx, BLSH_EINVAL, "misaligned pointer");
    if (N == 0) return BLSH_OK;
    blsh_device_guard g(ctx->device);
    return srp_sparse_cols(ctx, indptr, indices, values, N, Rq, dim, bits, col_begin, col_count, row_mask,
                                      sig, blsh_stream(stream));
}

extern "C" int blsh_srp_sparse_q16(blsh_ctx *ctx, const int64_t *indptr, const uint32_t *indices,
                                   const float *values, int64_t N, const uint16_t *Rq, int64_t dim, int32_t bits,
                                   uint32_t *sig, void *stream) {
    if (!ctx) return BLSH_EINVAL;
    if (!indptr || !indices || !values || !Rq || !sig)
        return blsh_fail(ctx, BLSH_EINVAL, "indptr, indices, values, Rq and sig are required");
    if (N < 0 || N >= (1ll << 32) || dim <= 0 || bits <= 0 || bits % 32 || bits > 4096)
        return blsh_fail(ctx, BLSH_EINVAL, "bits must be a positive multiple of 32, at most 4096; N < 2^32");
    if (!blsh_aligned(indptr, 8) || !blsh_aligned(Rq, 2)) return blsh_fail(ctx, BLSH_EINVAL, "misaligned pointer");
    if (N == 0) return BLSH_OK;
    blsh_device_guard g(ctx->device);
    cudaStream_t s = blsh_stream(stream);
    const long long cap = (long long)ctx->sm_count * 32;
    const unsigned grid = (unsigned)(N < cap ? N : cap);
    if (bits % 128 == 0 && blsh_aligned(Rq, 8))   // 8-byte loads of four codes
        return srp_sparse_cols(ctx, indptr, indices, values, N, Rq, dim, bits, 0, bits, nullptr, sig, s);
    int per_thread;
    const int T = srp_threads(bits, &per_thread);
    if (per_thread > kSrpMaxPerThread) return blsh_fail(ctx, BLSH_EINVAL, "bits/32 needs a divisor in 2..8");
    blsh_time_start(ctx, s);
    srp_sparse_kernel<uint16_t><<<grid, T, 0, s>>>(indptr, indices, values, N, Rq, dim, bits, per_thread, sig,
                                                   ctx->scratch);
    BLSH_LAUNCHED(ctx, "srp_sparse_kernel");
    return BLSH_OK;
}
