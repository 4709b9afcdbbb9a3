// allpairs.cu -- candidate generation by prefix filtering: the AllPairs
// method (Bayardo, Ma and Srikant, "Scaling up all pairs similarity search",
// WWW 2007), which Section 5.1 pairs with BayesLSH as the other source of
// candidates besides LSH.
//
//   1. feature statistics: document frequency df_f and the largest |weight|
//      maxabs_f of every feature (atomics over the nonzeros);
//   2. every row's indexed features.  Walking the row in the global order
//      (decreasing df, then increasing id), a running bound grows by
//      w_e = rn(|x_e| maxabs_f 2^48) (cosine; an exact integer sum, so the
//      order of the additions does not matter) or by 1 (sets); a feature is
//      indexed once the bound including it reaches the row's threshold
//      (cosine: ceil((t - 1e-9) 2^48); sets: ceil(t |x| - 1e-9)).  The
//      unindexed prefix then cannot lift a similarity to t, so every pair that
//      reaches t shares an indexed feature of its first row.  Rows of up to
//      128 elements: a warp, each element's bound the sum over the elements
//      that precede or equal it (one broadcast read of shared memory each); up
//      to 4096: a CTA sorts (order key, position) in shared memory and scans;
//      longer rows index every feature;
//   3. the inverted index: a key (feature, row) per indexed nonzero (padding
//      for the others), radix-sorted, so that a feature's list holds its rows
//      in increasing order, and each feature's list bounds from a scan of the
//      per-feature counts;
//   4. candidates: for every row y and feature f of y, the rows x < y of f's
//      list (a prefix of it, found by binary search) give the keys
//      (x << 32) | y: a count pass, an exclusive scan, a write pass (a warp
//      writes each prefix with coalesced stores);
//   5. the keys are radix-sorted, and the distinct ones are written as pairs
//      (x, y) in increasing order.
//
// Where N^2 <= 4096 max_dups and N^2 <= 2^31 + 512 max_dups (and N <= 2^19)
// steps 3 to 5 need no sort: the
// rows of every feature are listed in any order, and a CTA per row x sets bit
// y of an N-bit map in shared memory for every y > x in the lists of x's
// indexed features; the map's set bits, in order, are x's candidates (counted
// first, then written at scanned offsets; the write pass reads the counted maps
// again where N^2 / 8 bytes fit the place of the key buffers).  20,000 tf-idf
// rows (2.4e7 keys, 1.7e7 pairs): 1.96 ms by sorting, 0.37 ms with the maps.
// The line: a row's map of N / 32 words takes 0.4 ps a word to count and, not
// kept, 1.3 to 2.1 ps to form and write again; the sort takes about 50 ps a key
// of max_dups and 0.2 ms of launches.  Rows of 10 features, maps / sort:
// 8,000 rows, 1.6e4 keys 0.11 / 0.24 ms; 60,000, 9e5 0.46 / 0.45; 250,000,
// 1.6e7 3.5 / 1.5; 500,000, 6.3e7 20 / 4.0; 500,000, 6.3e8 26 / 27.
#include <type_traits>

#include "common.cuh"
#include "radix.cuh"
#include "scan.cuh"

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kShortRow = 128;
constexpr int kLongRow = 4096;
constexpr long long kMapRows = 1ll << 19;   // bit maps of up to 64 KB
// A count-only call walks the lists where every element's list of every row
// (nnz N entries, a bound known on the host) has at most 2^28 entries, else it
// sorts the index and searches it, whose time does not grow with the keys.  Rows
// that share nearly every feature, lists / sort: 2^27.2 entries 165 / 264 us,
// 2^28.3 233 / 274 and 164 / 158, 2^30.9 734 / 346.  (Always by lists: 250,000
// tf-idf rows 8.8 ms, sorted 2.5; between, where the lists are far shorter than
// their bound, the sort costs up to twice the time: 20,000 rows 288 / 415.)
constexpr double kListReads = 268435456.0;
constexpr double kTwo48 = 281474976710656.0;
constexpr long long kTermCap = 1ll << 50;

struct ApArgs {
    const int64_t *indptr;
    const uint32_t *indices;
    const float *values;    // NULL for sets
    long long N, dim;
    int cosine;
    double t;
    long long thr;          // cosine threshold in units of 2^-48
    uint32_t *df, *maxabs;  // [dim]: document frequency, largest |weight| (float bits)
    uint8_t *indexed;       // [nnz]
    blsh_dev_scratch *scratch;
};

// rn(|x| maxabs 2^48), capped (the cap lies far above any threshold, so it
// changes no decision and keeps the sums of a row below 2^63)
__device__ __forceinline__ long long ap_weight(const ApArgs &A, long long e, uint32_t f) {
    if (!A.cosine) return 1;
    const double p = __dmul_rn(__dmul_rn((double)fabsf(__ldg(A.values + e)), (double)__uint_as_float(A.maxabs[f])),
                               kTwo48);
    const long long w = __double2ll_rn(p);
    return w > kTermCap ? kTermCap : w;
}

// Threshold of a row of n elements: the bound value from which features are
// indexed (sets: ceil(t n - 1e-9) elements, formed in FP64 exactly as the
// oracle forms it).
__device__ __forceinline__ long long ap_threshold(const ApArgs &A, long long n) {
    if (A.cosine) return A.thr;
    return (long long)ceil(__dadd_rn(__dmul_rn(A.t, (double)n), -1e-9));
}

// Order key: decreasing df, then increasing id (ascending key order).
__device__ __forceinline__ unsigned long long ap_key(const ApArgs &A, uint32_t f) {
    return ((unsigned long long)(0xffffffffu - A.df[f]) << 32) | f;
}

// The elements of the rows: those before indptr[0] or past indptr[N] (some
// rows of a larger CSR) are no row's, so nothing counts them.
__device__ __forceinline__ void ap_elements(const ApArgs &A, long long nnz, long long &s, long long &e) {
    s = __ldg(A.indptr);
    e = min(nnz, (long long)__ldg(A.indptr + A.N));
}

// df and max |value| of every feature; with `place`, also each element's number
// among its feature's (in no particular order: where ap_post_kernel puts it, so
// the elements counted are those it places, and every entry is filled).
// Bound by the atomics on the most frequent features' addresses (20,000 rows:
// one feature stands in most of them); the largest value is looked at before
// it is replaced, and the numbers save ap_post_kernel the same atomics again
// (20,000 rows, 1.15e6 elements: 35 us and 51 us, now 46 and 19: an
// atomic whose answer is waited for costs more, two of them most).
__global__ void __launch_bounds__(256) ap_stats_kernel(ApArgs A, long long nnz, uint32_t *place) {
    unsigned long long bad = 0;
    long long s, end;
    ap_elements(A, nnz, s, end);
    for (long long e = s + (long long)blockIdx.x * blockDim.x + threadIdx.x; e < end; e += (long long)gridDim.x * blockDim.x) {
        const uint32_t f = __ldg(A.indices + e);
        if (f >= A.dim) { ++bad; continue; }
        const uint32_t at = atomicAdd(&A.df[f], 1u);
        if (place) place[e] = at;
        if (A.cosine) {
            const uint32_t v = __float_as_uint(fabsf(__ldg(A.values + e)));
            if (v > __ldcg(&A.maxabs[f])) atomicMax(&A.maxabs[f], v);
        }
    }
    if (bad) blsh_dev_error(A.scratch, BLSH_ERANGE, 0, bad);
}

// Rows of up to kShortRow elements (one warp per row, up to kShortRow / 32
// elements a lane) and rows longer than kLongRow (every feature indexed); the
// rows in between are listed for ap_prefix_cta_kernel (at most nnz / 129 of
// them).  The bound at an element
// is the sum of the weights that precede it in the global order and its own:
// n^2 comparisons, which a warp does faster than a CTA sorts while n <= 128
// (20,000 rows, mean 57: 208 us with a CTA for every row above 32 elements,
// 47 and 56 us with this).
__global__ void __launch_bounds__(256) ap_prefix_warp_kernel(ApArgs A, uint32_t *mid, unsigned *n_mid) {
    __shared__ ulonglong2 s_kw[8][kShortRow];   // order key, weight
    constexpr int EPL = kShortRow / 32;
    const int lane = threadIdx.x & 31;
    ulonglong2 *kw = s_kw[threadIdx.x >> 5];
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long row = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < A.N; row += nw) {
        const long long s = __ldg(A.indptr + row), n = __ldg(A.indptr + row + 1) - s;
        if (n > kLongRow) {
            for (long long i = lane; i < n; i += 32) A.indexed[s + i] = 1;
            continue;
        }
        if (n > kShortRow) {
            if (lane == 0) mid[atomicAdd(n_mid, 1u)] = (uint32_t)row;   // for ap_prefix_cta_kernel
            continue;
        }
        if (n == 0) continue;
        unsigned long long key[EPL];
        long long b[EPL];
        __syncwarp();                              // the previous row has been read
#pragma unroll
        for (int u = 0; u < EPL; ++u) {
            const int i = lane + 32 * u;
            key[u] = ~0ull;
            b[u] = 0;
            long long w = 0;
            if (i < n) {
                const uint32_t f = __ldg(A.indices + s + i);
                if (f < A.dim) {
                    key[u] = ap_key(A, f);
                    w = ap_weight(A, s + i, f);
                }
                kw[i] = make_ulonglong2(key[u], (unsigned long long)w);
            }
        }
        __syncwarp();
        auto sums = [&](auto used) {               // elements per lane that the row fills
            constexpr int U = decltype(used)::value;
#pragma unroll 4
            for (int j = 0; j < (int)n; ++j) {
                const ulonglong2 v = kw[j];
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (v.x <= key[u]) b[u] += (long long)v.y;
            }
        };
        if (n <= 32) sums(std::integral_constant<int, 1>{});
        else if (n <= 64) sums(std::integral_constant<int, 2>{});
        else sums(std::integral_constant<int, EPL>{});
        const long long thr = ap_threshold(A, n);
#pragma unroll
        for (int u = 0; u < EPL; ++u)
            if (lane + 32 * u < n) A.indexed[s + lane + 32 * u] = b[u] >= thr;
    }
}

// Rows of kShortRow+1 .. kLongRow elements, one CTA per row: (key, position)
// sorted in shared memory (bitonic), the weights scanned in that order.
constexpr int kCtaThreads = 256;
__global__ void __launch_bounds__(kCtaThreads) ap_prefix_cta_kernel(ApArgs A, const uint32_t *mid,
                                                                     const unsigned *n_mid) {
    __shared__ unsigned long long s_key[kLongRow];
    __shared__ uint16_t s_pos[kLongRow];
    __shared__ long long s_part[kCtaThreads / 32];
    const unsigned rows = *n_mid;
    for (unsigned q = blockIdx.x; q < rows; q += gridDim.x) {
        const long long row = mid[q];
        const long long s = __ldg(A.indptr + row), n = __ldg(A.indptr + row + 1) - s;
        int m = 1;
        while (m < n) m <<= 1;
        __syncthreads();
        for (int i = threadIdx.x; i < m; i += blockDim.x) {
            unsigned long long k = ~0ull;
            if (i < n) {
                const uint32_t f = __ldg(A.indices + s + i);
                if (f < A.dim) k = ap_key(A, f);
            }
            s_key[i] = k;
            s_pos[i] = (uint16_t)i;
        }
        __syncthreads();
        for (int size = 2; size <= m; size <<= 1)
            for (int stride = size >> 1; stride > 0; stride >>= 1) {
                for (int i = threadIdx.x; i < m; i += blockDim.x) {
                    const int p = i ^ stride;
                    if (p > i) {
                        const bool up = (i & size) == 0;
                        const unsigned long long a = s_key[i], b = s_key[p];
                        if ((a > b) == up) {
                            s_key[i] = b;
                            s_key[p] = a;
                            const uint16_t t = s_pos[i];
                            s_pos[i] = s_pos[p];
                            s_pos[p] = t;
                        }
                    }
                }
                __syncthreads();
            }
        // inclusive scan of the weights in sorted order, kCtaThreads at a time
        const long long thr = ap_threshold(A, n);
        long long carry = 0;
        for (int c0 = 0; c0 < n; c0 += blockDim.x) {
            const int i = c0 + threadIdx.x;
            long long w = 0;
            int pos = 0;
            if (i < n) {
                pos = s_pos[i];
                const uint32_t f = __ldg(A.indices + s + pos);
                w = f < A.dim ? ap_weight(A, s + pos, f) : 0;
            }
            long long x = w;
            const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long long y = __shfl_up_sync(kFull, x, o);
                if (lane >= o) x += y;
            }
            if (lane == 31) s_part[wid] = x;
            __syncthreads();
            long long before = carry;
            for (int q = 0; q < wid; ++q) before += s_part[q];
            long long total = carry;
            for (int q = 0; q < (int)(blockDim.x >> 5); ++q) total += s_part[q];
            if (i < n) A.indexed[s + pos] = before + x >= thr;
            __syncthreads();
            carry = total;
        }
    }
}

// Index keys: (feature << xbits) | row for indexed nonzeros, the padding key
// (all ones) for the others and for elements of no row; per-feature counts of
// indexed nonzeros.
__global__ void __launch_bounds__(256) ap_index_keys_kernel(ApArgs A, long long nnz, int xbits,
                                                            unsigned long long *keys, unsigned long long *fcnt) {
    const int lane = threadIdx.x & 31;
    {
        const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x, nt = (long long)gridDim.x * blockDim.x;
        long long first, end;
        ap_elements(A, nnz, first, end);
        for (long long i = t; i < first && i < nnz; i += nt) keys[i] = ~0ull;
        for (long long i = end + t; i < nnz; i += nt) keys[i] = ~0ull;
    }
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long row = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < A.N; row += nw) {
        const long long s = __ldg(A.indptr + row), e = __ldg(A.indptr + row + 1);
        for (long long i = s + lane; i < e; i += 32) {
            const uint32_t f = __ldg(A.indices + i);
            unsigned long long k = ~0ull;
            if (f < A.dim && A.indexed[i]) {
                k = ((unsigned long long)f << xbits) | (unsigned long long)row;
                atomicAdd(fcnt + f, 1ull);
            }
            keys[i] = k;
        }
    }
}

// First position in the sorted list L[0..n) (row ids in the low xbits of the
// keys) whose row is >= y.
__device__ __forceinline__ long long ap_lower(const unsigned long long *L, long long n, uint32_t y,
                                              unsigned long long xmask) {
    long long lo = 0, hi = n;
    while (lo < hi) {
        const long long mid = (lo + hi) >> 1;
        if ((uint32_t)(__ldg(L + mid) & xmask) < y) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// Count pass (WRITE = false): ycnt[y] = sum over the features f of row y of
// the number of rows x < y in f's list.  Write pass: the keys (x << 32) | y at
// offsets ycnt[y] (after the scan), at most cap of them.
template <bool WRITE>
__global__ void __launch_bounds__(256) ap_emit_kernel(ApArgs A, const unsigned long long *ikeys,
                                                      const unsigned long long *fstart, unsigned long long xmask,
                                                      unsigned long long *ycnt, unsigned long long *out,
                                                      long long cap) {
    const int lane = threadIdx.x & 31;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long y = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; y < A.N; y += nw) {
        const long long s = __ldg(A.indptr + y), e = __ldg(A.indptr + y + 1);
        unsigned long long base = WRITE ? ycnt[y] : 0ull;
        unsigned long long total = 0;
        for (long long c0 = s; c0 < e; c0 += 32) {
            long long lo = 0, cnt = 0;
            if (c0 + lane < e) {
                const uint32_t f = __ldg(A.indices + c0 + lane);
                if (f < A.dim) {
                    lo = (long long)fstart[f];
                    cnt = ap_lower(ikeys + lo, (long long)(fstart[f + 1] - fstart[f]), (uint32_t)y, xmask);
                }
            }
            if (!WRITE) {
                total += (unsigned long long)cnt;
                continue;
            }
            // offsets of this chunk's prefixes, then each written by the whole warp
            long long incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long long v = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += v;
            }
            const long long excl = incl - cnt;
            for (int l = 0; l < 32; ++l) {
                const long long n_l = __shfl_sync(kFull, cnt, l);
                if (n_l == 0) continue;
                const long long lo_l = __shfl_sync(kFull, lo, l);
                const unsigned long long o_l = base + (unsigned long long)__shfl_sync(kFull, excl, l);
                for (long long i = lane; i < n_l; i += 32) {
                    const unsigned long long x = __ldg(ikeys + lo_l + i) & xmask;
                    if (o_l + (unsigned long long)i < (unsigned long long)cap)
                        out[o_l + i] = (x << 32) | (unsigned long long)y;
                }
            }
            base += (unsigned long long)__shfl_sync(kFull, incl, 31);
        }
        if (!WRITE) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(kFull, total, o);
            if (lane == 0) ycnt[y] = total;
        }
    }
}

// Keys from the total (device) up to cap get the padding key (sorted last).
__global__ void __launch_bounds__(256) ap_pad_kernel(unsigned long long *keys, const unsigned long long *total,
                                                     long long cap) {
    const long long n = (long long)*total;
    for (long long i = (n < 0 ? 0 : n) + (long long)blockIdx.x * blockDim.x + threadIdx.x; i < cap;
         i += (long long)gridDim.x * blockDim.x)
        keys[i] = ~0ull;
}

// Distinct-key marks: mark[i] = 1 where key i is not padding and differs
// from key i-1.
__global__ void __launch_bounds__(256) ap_mark_kernel(const unsigned long long *keys, long long n, uint32_t *mark) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const unsigned long long k = keys[i];
        mark[i] = k != ~0ull && (i == 0 || keys[i - 1] != k);
    }
}

// The distinct keys as pairs, at their scanned positions (at most cap).
__global__ void __launch_bounds__(256) ap_write_kernel(const unsigned long long *keys, const uint32_t *mark,
                                                       const uint32_t *pos, long long n, uint32_t *pairs, long long cap) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        if (!mark[i]) continue;
        const long long p = pos[i];
        if (p < cap) {
            pairs[2 * p] = (uint32_t)(keys[i] >> 32);
            pairs[2 * p + 1] = (uint32_t)keys[i];
        }
    }
}

// ---- candidates by bit maps ---------------------------------------------------

// Every feature's rows, in any order: post[fstart[f] .. fstart[f + 1]).
__global__ void __launch_bounds__(256) ap_post_kernel(ApArgs A, const uint32_t *fstart, const uint32_t *place,
                                                      uint32_t *post) {
    const int lane = threadIdx.x & 31;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long row = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < A.N; row += nw) {
        const long long s = __ldg(A.indptr + row), e = __ldg(A.indptr + row + 1);
        for (long long i = s + lane; i < e; i += 32) {
            const uint32_t f = __ldg(A.indices + i);
            if (f < A.dim) post[__ldg(fstart + f) + __ldg(place + i)] = (uint32_t)row;
        }
    }
}

// One CTA per row x, rows from a counter (the work of a row varies a hundredfold
// with its features' frequencies).  MAP_COUNT: cnt[x] = the number of distinct
// y > x in the lists of x's indexed features.  MAP_WRITE: the pairs (x, y), y
// increasing, from offset cnt[x] (after the scan).  Both MAP_COUNT and
// MAP_DUPS (which forms no map) add the number of (feature, y) met to
// *dup_total, the number of keys the sorting form would have.  With `kept`
// MAP_COUNT leaves every row's map there (word x words + i, words from that of
// x + 1 on) for ap_map_write_kernel.
enum { MAP_DUPS, MAP_COUNT, MAP_WRITE };
template <int MODE>
__global__ void __launch_bounds__(256) ap_map_kernel(ApArgs A, const uint32_t *fstart, const uint32_t *post,
                                                     unsigned long long *cnt, unsigned long long *dup_total,
                                                     long long max_dups, uint32_t *pairs, long long cap,
                                                     unsigned *next_row, uint32_t *kept) {
    extern __shared__ uint32_t map[];   // [(N + 31) / 32], zero between rows
    __shared__ unsigned s_cnt, s_row[2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (MODE == MAP_WRITE && (long long)*dup_total > max_dups) return;   // no pairs: the buffer was too small
    const int words = (int)((A.N + 31) >> 5);
    if (MODE != MAP_DUPS)
        for (int i = threadIdx.x; i < words; i += blockDim.x) map[i] = 0;
    if (threadIdx.x == 0) s_cnt = 0;
    unsigned long long dups = 0;
    for (int turn = 0;; turn ^= 1) {
        if (threadIdx.x == 0) s_row[turn] = atomicAdd(next_row, 1u);
        __syncthreads();                         // the row is there, the map is clear
        const uint32_t x = s_row[turn];          // N < 2^31
        if (x >= A.N) break;
        const long long s = __ldg(A.indptr + x), e = __ldg(A.indptr + x + 1);
        // 32 features' list bounds at a time, one per lane (so that their
        // dependent loads overlap); each warp walks every eighth list, four
        // loads in flight
        for (long long i0 = s; i0 < e; i0 += 32) {
            uint32_t l0 = 0, l1 = 0;
            if (i0 + lane < e && A.indexed[i0 + lane]) {
                const uint32_t f = __ldg(A.indices + i0 + lane);
                if (f < A.dim) {
                    l0 = __ldg(fstart + f);
                    l1 = __ldg(fstart + f + 1);
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t begin = __shfl_sync(kFull, l0, 8 * q + warp), end = __shfl_sync(kFull, l1, 8 * q + warp);
                for (uint32_t l = begin + lane; l < end + lane; l += 128) {   // (warp-uniform trip count)
                    uint32_t y[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) y[k] = l + 32 * k < end ? __ldg(post + l + 32 * k) : 0u;
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (y[k] > x) {
                            if (MODE != MAP_DUPS) atomicOr(map + (y[k] >> 5), 1u << (y[k] & 31));
                            ++dups;
                        }
                }
            }
        }
        if (MODE == MAP_DUPS) continue;
        __syncthreads();
        const int w0 = (int)((x + 1) >> 5);
        if (MODE == MAP_COUNT) {
            unsigned c = 0;
            for (int i = w0 + threadIdx.x; i < words; i += blockDim.x) {
                const uint32_t m = map[i];
                c += __popc(m);
                map[i] = 0;
                if (kept) kept[(size_t)x * words + i] = m;
            }
            c = __reduce_add_sync(kFull, c);
            if (lane == 0 && c) atomicAdd(&s_cnt, c);
            __syncthreads();
            if (threadIdx.x == 0) {
                cnt[x] = s_cnt;
                s_cnt = 0;
            }
        } else {
            long long base = (long long)cnt[x];
            const long long end = (long long)cnt[x + 1];
            for (int i0 = w0; i0 < words && base < end; i0 += blockDim.x) {
                const int i = i0 + threadIdx.x;
                uint32_t m = 0;
                if (i < words) {
                    m = map[i];
                    map[i] = 0;
                }
                unsigned total;
                long long o = base + blsh_scan::block_exclusive<unsigned>((unsigned)__popc(m), &total);
                base += total;
                for (; m; m &= m - 1, ++o)
                    if (o < cap) reinterpret_cast<uint2 *>(pairs)[o] = make_uint2(x, 32u * i + __ffs(m) - 1u);
            }
        }
    }
    if (MODE != MAP_WRITE) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) dups += __shfl_xor_sync(kFull, dups, o);
        if (lane == 0 && dups) atomicAdd(dup_total, dups);
    }
}

// The pairs of the kept maps: a warp per row, 32 words at a time, put in order in
// shared memory so that they leave in coalesced stores.  20,000 rows, 1.6e7
// pairs: MAP_WRITE, which forms every map again, 172 us, 49 here.
constexpr int kKeptWarps = 8;
__global__ void __launch_bounds__(32 * kKeptWarps) ap_map_write_kernel(long long N, const uint32_t *kept,
                                                                       const unsigned long long *cnt,
                                                                       const unsigned long long *dup_total,
                                                                       long long max_dups, uint32_t *pairs,
                                                                       long long cap) {
    __shared__ uint32_t s_y[kKeptWarps][1024];
    if ((long long)*dup_total > max_dups) return;   // no pairs: the buffer was too small
    const int lane = threadIdx.x & 31;
    uint32_t *ys = s_y[threadIdx.x >> 5];
    const int words = (int)((N + 31) >> 5);
    const long long nw = (long long)gridDim.x * kKeptWarps;
    for (long long x = (long long)blockIdx.x * kKeptWarps + (threadIdx.x >> 5); x < N; x += nw) {
        long long base = (long long)cnt[x];
        const long long end = (long long)cnt[x + 1];
        const uint32_t *row = kept + (size_t)x * words;
        int i = (int)((x + 1) >> 5) + lane;
        uint32_t next = i < words && base < end ? __ldcs(row + i) : 0u;
        for (; base < end; i += 32) {
            const uint32_t m = next;
            next = i + 32 < words ? __ldcs(row + i + 32) : 0u;
            const int c = __popc(m);
            int incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += v;
            }
            const int total = __shfl_sync(kFull, incl, 31);
            int at = incl - c;
            for (uint32_t b = m; b; b &= b - 1) ys[at++] = 32u * i + __ffs(b) - 1u;
            __syncwarp();
            for (int k = lane; k < total; k += 32)
                if (base + k < cap) reinterpret_cast<uint2 *>(pairs)[base + k] = make_uint2((uint32_t)x, ys[k]);
            __syncwarp();
            base += total;
        }
    }
}

// n_pairs = the number of distinct keys; truncation and an undersized key
// buffer are reported on the device.
template <typename T>
__global__ void ap_finish_kernel(const T *mark_total, const unsigned long long *dup_total, long long dup_cap,
                                 long long cap, int64_t *n_pairs, int64_t *n_dups, blsh_dev_scratch *scratch) {
    const long long dups = (long long)*dup_total;
    if (n_dups) *n_dups = dups;
    if (dups > dup_cap) {   // the key buffer was too small: no pairs
        *n_pairs = 0;
        blsh_dev_error(scratch, BLSH_ETRUNC, 1, (unsigned long long)(dups - dup_cap));
        return;
    }
    const long long n = (long long)*mark_total;
    *n_pairs = n;
    if (n > cap) blsh_dev_error(scratch, BLSH_ETRUNC, 1, (unsigned long long)(n - cap));
}

// Count-only calls: n_dups and n_pairs = 0 (the pairs are not formed).
__global__ void ap_count_only_kernel(const unsigned long long *dup_total, int64_t *n_pairs, int64_t *n_dups) {
    if (n_dups) *n_dups = (long long)*dup_total;
    *n_pairs = 0;
}

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

struct ApLayout {
    size_t df, maxabs, indexed, ik0, ik1, iv0, iv1, fcnt, ycnt, k0, k1, v0, v1, mark, pos, hist, partial, grand,
        total;
};

ApLayout ap_layout(long long N, long long nnz, long long dim, long long max_dups) {
    const long long big = nnz > max_dups ? nnz : max_dups;
    const long long scan_n = (N + 1 > dim + 1 ? N + 1 : dim + 1) > big ? (N + 1 > dim + 1 ? N + 1 : dim + 1) : big;
    ApLayout L;
    size_t o = 0;
    L.df = o; o = up256(o + dim * 4);
    L.maxabs = o; o = up256(o + dim * 4);
    L.indexed = o; o = up256(o + nnz);
    L.ik0 = o; o = up256(o + nnz * 8);
    L.ik1 = o; o = up256(o + nnz * 8);
    L.iv0 = o; o = up256(o + nnz * 4);
    L.iv1 = o; o = up256(o + nnz * 4);
    L.fcnt = o; o = up256(o + (dim + 1) * 8);
    L.ycnt = o; o = up256(o + (N + 1) * 8);
    L.k0 = o; o = up256(o + max_dups * 8);
    L.k1 = o; o = up256(o + max_dups * 8);
    L.v0 = o; o = up256(o + max_dups * 4);
    L.v1 = o; o = up256(o + max_dups * 4);
    L.mark = o; o = up256(o + max_dups * 4);
    L.pos = o; o = up256(o + max_dups * 4);
    L.hist = o; o = up256(o + blsh_radix::hist_entries(big) * 4);
    const long long part = blsh_radix::partial_entries(big) + blsh_scan::tiles_for(scan_n) + 2;
    L.partial = o; o = up256(o + part * 8);
    L.grand = o; o = up256(o + 64);
    L.total = o;
    return L;
}

int bits_for(long long v) {
    int b = 1;
    while (b < 63 && (1ll << b) <= v) ++b;
    return b;
}

}  // namespace

extern "C" int blsh_allpairs_workspace(int64_t N, int64_t nnz, int64_t dim, int64_t max_dups, size_t *bytes) {
    if (!bytes || N < 0 || nnz < 0 || dim <= 0 || max_dups < 0) return BLSH_EINVAL;
    *bytes = ap_layout(N, nnz, dim, max_dups).total;
    return BLSH_OK;
}

extern "C" int blsh_allpairs_candidates(blsh_ctx *ctx, const int64_t *indptr, const uint32_t *indices,
                                        const float *values, int64_t N, int64_t nnz, int64_t dim, double t,
                                        int32_t kind,
                                        int64_t max_dups, uint32_t *pairs, int64_t cap, int64_t *n_pairs,
                                        int64_t *n_dups, void *workspace, size_t workspace_bytes, void *stream) {
    if (!ctx) return BLSH_EINVAL;
    if (!indptr || !n_pairs || (N > 0 && !indices) || (cap > 0 && !pairs))
        return blsh_fail(ctx, BLSH_EINVAL, "indptr, indices and n_pairs are required");
    if (kind != BLSH_JACCARD && kind != BLSH_COSINE) return blsh_fail(ctx, BLSH_EINVAL, "bad kind");
    if ((kind == BLSH_COSINE) != (values != nullptr))
        return blsh_fail(ctx, BLSH_EINVAL, "values must be given for cosine rows and only for them");
    if (!(t > 0 && t < 1)) return blsh_fail(ctx, BLSH_EINVAL, "t must lie in (0, 1)");
    if (N < 0 || N >= (1ll << 32) || dim <= 0 || dim > (1ll << 32) || cap < 0 || max_dups < 0 || max_dups >= (1ll << 32))
        return blsh_fail(ctx, BLSH_EINVAL, "bad N, dim, cap or max_dups");
    if (!blsh_aligned(indptr, 8) || !blsh_aligned(n_pairs, 8) || !blsh_aligned(n_dups, 8) ||
        !blsh_aligned(workspace, 256) || !blsh_aligned(pairs, 8))
        return blsh_fail(ctx, BLSH_EINVAL, "misaligned pointer");
    blsh_device_guard g(ctx->device);
    cudaStream_t s = blsh_stream(stream);
    if (N < 2) {
        BLSH_CUDA(ctx, cudaMemsetAsync(n_pairs, 0, sizeof(int64_t), s));
        if (n_dups) BLSH_CUDA(ctx, cudaMemsetAsync(n_dups, 0, sizeof(int64_t), s));
        return BLSH_OK;
    }
    if (nnz < 0 || nnz >= (1ll << 32)) return blsh_fail(ctx, BLSH_EINVAL, "nnz must lie in [0, 2^32)");
    const long long dcap = cap > 0 ? max_dups : 0;   // a count-only call needs no key buffers
    const ApLayout L = ap_layout(N, nnz, dim, dcap);
    if (!workspace || workspace_bytes < L.total) return blsh_fail(ctx, BLSH_ETRUNC, "workspace needs %zu bytes", L.total);
    char *ws = (char *)workspace;
    ApArgs A;
    A.indptr = indptr;
    A.indices = indices;
    A.values = values;
    A.N = N;
    A.dim = dim;
    A.cosine = kind == BLSH_COSINE;
    A.t = t;
    A.thr = (long long)ceil((t - 1e-9) * kTwo48);
    A.df = (uint32_t *)(ws + L.df);
    A.maxabs = (uint32_t *)(ws + L.maxabs);
    A.indexed = (uint8_t *)(ws + L.indexed);
    A.scratch = ctx->scratch;
    unsigned long long *fcnt = (unsigned long long *)(ws + L.fcnt);
    unsigned long long *ycnt = (unsigned long long *)(ws + L.ycnt);
    uint32_t *hist = (uint32_t *)(ws + L.hist);
    unsigned long long *partial64 = (unsigned long long *)(ws + L.partial);
    unsigned long long *grand64 = (unsigned long long *)(ws + L.grand);
    uint32_t *grand32 = (uint32_t *)(ws + L.grand + 16);
    unsigned long long *dup_total = (unsigned long long *)(ws + L.grand + 32);
    const int sms = ctx->sm_count;
    auto grid_for = [&](long long items, long long per_block) {
        const long long b = (items + per_block - 1) / per_block, cap_b = (long long)sms * 16;
        return (unsigned)(b < 1 ? 1 : (b < cap_b ? b : cap_b));
    };

    // 1. statistics
    BLSH_CUDA(ctx, cudaMemsetAsync(A.df, 0, L.indexed - L.df, s));   // df and maxabs
    BLSH_CUDA(ctx, cudaMemsetAsync(ws + L.grand, 0, 64, s));         // the totals and counters
    // bit maps where they cost less than sorting the keys (see the top of the
    // file); a count-only call forms neither map nor key, and walks the lists
    // only where all of them for every element are few
    const bool count_only = cap == 0 || max_dups == 0;
    const bool maps = N <= kMapRows && nnz < (1ll << 31) &&
                      (count_only ? (double)nnz * (double)N <= kListReads
                                  : N * N <= 4096 * max_dups && N * N <= (1ll << 31) + 512 * max_dups);
    uint32_t *place = (uint32_t *)(ws + L.iv0);
    blsh_time_start(ctx, s);
    ap_stats_kernel<<<grid_for(nnz, 256), 256, 0, s>>>(A, nnz, maps ? place : nullptr);
    BLSH_LAUNCHED(ctx, "ap_stats_kernel");
    // 2. indexed features
    blsh_time_start(ctx, s);
    uint32_t *mid = (uint32_t *)(ws + L.ik1);                 // rows of 129 .. 4,096 elements
    unsigned *n_mid = (unsigned *)(ws + L.grand + 48);
    ap_prefix_warp_kernel<<<grid_for(N, 8), 256, 0, s>>>(A, mid, n_mid);
    BLSH_LAUNCHED(ctx, "ap_prefix_warp_kernel");
    blsh_time_start(ctx, s);
    ap_prefix_cta_kernel<<<(unsigned)sms * 4, kCtaThreads, 0, s>>>(A, mid, n_mid);
    BLSH_LAUNCHED(ctx, "ap_prefix_cta_kernel");
    if (maps) {
        uint32_t *fstart = (uint32_t *)(ws + L.fcnt), *post = (uint32_t *)(ws + L.ik0);
        if (const int rc = blsh_scan::run<uint32_t>(ctx, A.df, fstart, dim, (uint32_t *)partial64, fstart + dim, s)) return rc;
        blsh_time_start(ctx, s);
        ap_post_kernel<<<grid_for(N, 8), 256, 0, s>>>(A, fstart, place, post);
        BLSH_LAUNCHED(ctx, "ap_post_kernel");
        const unsigned grid = (unsigned)(N < (long long)sms * 8 ? N : (long long)sms * 8);
        if (count_only) {
            blsh_time_start(ctx, s);
            ap_map_kernel<MAP_DUPS><<<grid, 256, 0, s>>>(A, fstart, post, nullptr, dup_total, 0, nullptr, 0,
                                                                n_mid + 1, nullptr);
            BLSH_LAUNCHED(ctx, "ap_map_kernel (keys)");
            ap_count_only_kernel<<<1, 1, 0, s>>>(dup_total, n_pairs, n_dups);
            BLSH_LAUNCHED(ctx, "ap_count_only_kernel");
            return BLSH_OK;
        }
        const size_t smem = (size_t)((N + 31) / 32) * 4;
        // (always: the launch default of 48 KB holds a kernel's own shared memory too)
        BLSH_CUDA(ctx, cudaFuncSetAttribute(ap_map_kernel<MAP_COUNT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)(kMapRows / 8)));
        BLSH_CUDA(ctx, cudaFuncSetAttribute(ap_map_kernel<MAP_WRITE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)(kMapRows / 8)));
        // the maps are kept for the write pass where they fit the key buffers' place (N^2 / 8 of 32 max_dups bytes)
        uint32_t *kept = (size_t)N * smem <= L.hist - L.k0 ? (uint32_t *)(ws + L.k0) : nullptr;
        blsh_time_start(ctx, s);
        ap_map_kernel<MAP_COUNT><<<grid, 256, smem, s>>>(A, fstart, post, ycnt, dup_total, max_dups, nullptr, 0,
                                                             n_mid + 1, kept);
        BLSH_LAUNCHED(ctx, "ap_map_kernel (count pass)");
        if (const int rc = blsh_scan::run<unsigned long long>(ctx, ycnt, ycnt, N, partial64, ycnt + N, s)) return rc;
        blsh_time_start(ctx, s);
        if (kept)
            ap_map_write_kernel<<<grid_for(N, kKeptWarps), 32 * kKeptWarps, 0, s>>>(N, kept, ycnt, dup_total, max_dups,
                                                                                     pairs, cap);
        else
            ap_map_kernel<MAP_WRITE><<<grid, 256, smem, s>>>(A, fstart, post, ycnt, dup_total, max_dups, pairs, cap,
                                                             n_mid + 2, nullptr);
        BLSH_LAUNCHED(ctx, "ap_map_kernel (write pass)");
        ap_finish_kernel<<<1, 1, 0, s>>>(ycnt + N, dup_total, max_dups, cap, n_pairs, n_dups, ctx->scratch);
        BLSH_LAUNCHED(ctx, "ap_finish_kernel");
        return BLSH_OK;
    }
    // 3. the inverted index
    const int xbits = bits_for(N);
    const int key_bits = xbits + bits_for(dim);
    unsigned long long *ik[2] = {(unsigned long long *)(ws + L.ik0), (unsigned long long *)(ws + L.ik1)};
    uint32_t *iv[2] = {(uint32_t *)(ws + L.iv0), (uint32_t *)(ws + L.iv1)};
    BLSH_CUDA(ctx, cudaMemsetAsync(fcnt, 0, (dim + 1) * 8, s));
    blsh_time_start(ctx, s);
    ap_index_keys_kernel<<<grid_for(N, 8), 256, 0, s>>>(A, nnz, xbits, ik[0], fcnt);
    BLSH_LAUNCHED(ctx, "ap_index_keys_kernel");
    int cur = 0;
    {
        // the padding key (all ones) sorts after every real key in key_bits bits
        const int rc = blsh_radix::sort(ctx, ik, iv, nnz, 64 > key_bits ? key_bits + 1 : 64, hist,
                                        (uint32_t *)partial64, grand32, s, &cur);
        if (rc) return rc;
    }
    // feature list starts: exclusive scan of the per-feature counts (dim + 1 entries)
    if (const int rc = blsh_scan::run<unsigned long long>(ctx, fcnt, fcnt, dim + 1, partial64, grand64, s)) return rc;
    const unsigned long long xmask = (1ull << xbits) - 1ull;
    // 4. candidate keys: count, scan, write
    blsh_time_start(ctx, s);
    ap_emit_kernel<false><<<grid_for(N, 8), 256, 0, s>>>(A, ik[cur], fcnt, xmask, ycnt, nullptr, 0);
    BLSH_LAUNCHED(ctx, "ap_emit_kernel (count pass)");
    BLSH_CUDA(ctx, cudaMemsetAsync(ycnt + N, 0, 8, s));
    if (const int rc = blsh_scan::run<unsigned long long>(ctx, ycnt, ycnt, N + 1, partial64, dup_total, s)) return rc;
    if (cap == 0 || max_dups == 0) {
        ap_count_only_kernel<<<1, 1, 0, s>>>(dup_total, n_pairs, n_dups);
        BLSH_LAUNCHED(ctx, "ap_count_only_kernel");
        return BLSH_OK;
    }
    unsigned long long *ck[2] = {(unsigned long long *)(ws + L.k0), (unsigned long long *)(ws + L.k1)};
    uint32_t *cv[2] = {(uint32_t *)(ws + L.v0), (uint32_t *)(ws + L.v1)};
    blsh_time_start(ctx, s);
    ap_emit_kernel<true><<<grid_for(N, 8), 256, 0, s>>>(A, ik[cur], fcnt, xmask, ycnt, ck[0], max_dups);
    BLSH_LAUNCHED(ctx, "ap_emit_kernel (write pass)");
    blsh_time_start(ctx, s);
    ap_pad_kernel<<<grid_for(max_dups, 256), 256, 0, s>>>(ck[0], dup_total, max_dups);
    BLSH_LAUNCHED(ctx, "ap_pad_kernel");
    // 5. sort, keep the distinct keys
    int kc = 0;
    {
        // keys (x << 32) | y: the write pass leaves them grouped by y in
        // increasing order, so a stable sort by x alone (bits 32 .. 32 + xbits,
        // one more bit for the padding key) orders them by (x, y)
        const int kbits = xbits + 1 < 32 ? xbits + 1 : 32;
        const int rc = blsh_radix::sort(ctx, ck, cv, max_dups, kbits, hist, (uint32_t *)partial64, grand32, s, &kc,
                                        32);
        if (rc) return rc;
    }
    uint32_t *mark = (uint32_t *)(ws + L.mark), *pos = (uint32_t *)(ws + L.pos);
    blsh_time_start(ctx, s);
    ap_mark_kernel<<<grid_for(max_dups, 256), 256, 0, s>>>(ck[kc], max_dups, mark);
    BLSH_LAUNCHED(ctx, "ap_mark_kernel");
    if (const int rc = blsh_scan::run<uint32_t>(ctx, mark, pos, max_dups, (uint32_t *)partial64, grand32, s)) return rc;
    blsh_time_start(ctx, s);
    ap_write_kernel<<<grid_for(max_dups, 256), 256, 0, s>>>(ck[kc], mark, pos, max_dups, pairs, cap);
    BLSH_LAUNCHED(ctx, "ap_write_kernel");
    ap_finish_kernel<<<1, 1, 0, s>>>(grand32, dup_total, max_dups, cap, n_pairs, n_dups, ctx->scratch);
    BLSH_LAUNCHED(ctx, "ap_finish_kernel");
    return BLSH_OK;
}
