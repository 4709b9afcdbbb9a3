// band.cu -- LSH banding candidate generation (Section 2, "Candidate
// generation via LSH"): objects whose `rows` hashes agree on a whole band
// become a candidate pair.
//
// The paper's hashtables are replaced by a sort:
//   1. every (band b, object i) gets a sort key: the band's hashes themselves
//      (cosine: the `rows` sign bits, exact) or bits of a 64-bit hash of them
//      (Jaccard);
//   2. an LSD radix sort (stable) groups equal keys within every band, objects
//      in increasing order inside a group;
//   3. for each sorted position p, the pairs (p, q > p) inside its group are
//      counted, then written at offsets from a prefix sum.  A pair is written
//      only for the first band in which it collides, so every distinct pair
//      appears once.  To find that band cheaply every object also has a row
//      of its band keys in band order: cosine keys packed as bytes, 16-bit
//      or 32-bit lanes (by `rows`; for 8, 16 and 32 rows that is the signature
//      row itself), compared by XOR and a zero-lane test; Jaccard class ids of
//      32 bits, or 64-bit band hashes confirmed by comparing the hashes
//      themselves, so a hash collision never merges buckets.  The count pass
//      records which pairs it keeps (one bit per tested pair, in the
//      workspace's keep record), and the write pass writes those pairs
//      without testing them again.
//
// The staged form (32-bit keys without the band index, warps over chunks of
// 32 sorted positions) takes cosine bands whose key rows fit 128 bytes and
// Jaccard up to 32 bands; emit_kernel and 64-bit keys take the rest.
#include <type_traits>

#include "common.cuh"
#include "radix.cuh"
#include "scan.cuh"

namespace {

constexpr unsigned kFull = 0xffffffffu;
using blsh_radix::kSortTile;

__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

// `rows` sign bits starting at bit `start` of a row (bit j in word j/32).
__device__ __forceinline__ uint32_t bit_field(const uint32_t *row, int start, int rows) {
    const int w = start >> 5, o = start & 31;
    unsigned long long two = __ldg(row + w);
    if (o + rows > 32) two |= (unsigned long long)__ldg(row + w + 1) << 32;
    const unsigned long long mask = rows == 32 ? 0xffffffffull : ((1ull << rows) - 1);
    return (uint32_t)((two >> o) & mask);
}

__device__ __forceinline__ unsigned long long band_hash(const uint32_t *row, int start, int rows) {
    unsigned long long h = 0x243f6a8885a308d3ull;
    for (int r = 0; r < rows; ++r) h = mix64(h ^ (__ldg(row + start + r) + 0x9e3779b97f4a7c15ull * (r + 1)));
    return h;
}

struct BandArgs {
    const uint32_t *sig;
    long long N;
    int W, kind, rows, bands, band_bits, key_shift;
    unsigned long long *bk;   // Jaccard: [N][bands] band hashes
    uint32_t *ck;             // cosine: [N][ck_words] band keys packed in lanes of ck_lane bytes
    int ck_lane, ck_words, ck_stride;   // words of a key row, and between the starts of two
    int vec16;                // rows of sig start 16-byte aligned
    int exact_classes;        // Jaccard: class ids in ck (4-byte lanes), 32-bit sort keys, no bk
};

// Lane width (bytes) of packed cosine band keys, and 32-bit words per row
// (rounded up to a multiple of 4 words so rows are 16-byte aligned).
__host__ __device__ inline int cos_lane_bytes(int rows) { return rows <= 8 ? 1 : (rows <= 16 ? 2 : 4); }
__host__ __device__ inline int cos_row_words(int rows, int bands) {
    const int words = (bands * cos_lane_bytes(rows) + 3) / 4;
    return (words + 3) & ~3;
}

__global__ void band_keys_kernel(BandArgs A, unsigned long long *keys, uint32_t *vals) {
    const long long n = A.N * A.bands;
    for (long long it = (long long)blockIdx.x * blockDim.x + threadIdx.x; it < n;
         it += (long long)gridDim.x * blockDim.x) {
        const int b = (int)(it / A.N);
        const long long i = it - (long long)b * A.N;
        const uint32_t *row = A.sig + (size_t)i * A.W;
        unsigned long long key;
        if (A.kind == BLSH_COSINE) {
            const uint32_t f = bit_field(row, b * A.rows, A.rows);
            key = ((unsigned long long)b << A.rows) | f;
            unsigned char *kr = reinterpret_cast<unsigned char *>(A.ck + (size_t)i * A.ck_words);
            if (A.ck_lane == 1) kr[b] = (unsigned char)f;
            else if (A.ck_lane == 2) reinterpret_cast<uint16_t *>(kr)[b] = (uint16_t)f;
            else reinterpret_cast<uint32_t *>(kr)[b] = f;
        } else {
            const unsigned long long h = band_hash(row, b * A.rows, A.rows);
            A.bk[(size_t)i * A.bands + b] = h;
            key = A.band_bits == 0 ? h : (((unsigned long long)b << A.key_shift) | (h >> A.band_bits));
        }
        keys[it] = key;
        vals[it] = (uint32_t)i;
    }
}

// ---- pair emission -----------------------------------------------------------

__device__ __forceinline__ bool same_band(const BandArgs &A, uint32_t x, uint32_t y, int b) {
    const uint32_t *rx = A.sig + (size_t)x * A.W, *ry = A.sig + (size_t)y * A.W;
    if (A.kind == BLSH_COSINE) return bit_field(rx, b * A.rows, A.rows) == bit_field(ry, b * A.rows, A.rows);
    const int start = b * A.rows;
    if (A.vec16 && (A.rows & 3) == 0 && (start & 3) == 0) {   // whole 16-byte groups
        const uint4 *vx = reinterpret_cast<const uint4 *>(rx + start), *vy = reinterpret_cast<const uint4 *>(ry + start);
        for (int r = 0; r < (A.rows >> 2); ++r) {
            const uint4 u = __ldg(vx + r), v = __ldg(vy + r);
            if (u.x != v.x || u.y != v.y || u.z != v.z || u.w != v.w) return false;
        }
        return true;
    }
    for (int r = 0; r < A.rows; ++r)
        if (__ldg(rx + start + r) != __ldg(ry + start + r)) return false;
    return true;
}

// Jaccard: the pair (x, y) met in band b is emitted iff b is the first band
// whose keys agree in full.  The 64-bit band hashes find the candidate bands
// (equal keys have equal hashes); a hash match is confirmed on the keys
// themselves before it decides anything.
__device__ __forceinline__ bool emit_here_jaccard(const BandArgs &A, uint32_t x, uint32_t y, int b) {
    const unsigned long long *bx = A.bk + (size_t)x * A.bands, *by = A.bk + (size_t)y * A.bands;
    for (int c = 0; c <= b; ++c)
        if (__ldg(bx + c) == __ldg(by + c) && same_band(A, x, y, c)) return c == b;
    return false;   // band b's hashes or keys differ: only a truncated-hash collision put them together
}

// Nonzero iff some lane of v (lanes of 1, 2 or 4 bytes) is zero.  The
// borrow of the subtraction can also flag a lane above a zero lane, never a
// lane below the lowest zero lane, so "any zero lane among the low lanes" is
// exact once the lanes above are masked off.
__device__ __forceinline__ uint32_t zero_lanes(uint32_t v, int lane) {
    if (lane == 1) return (v - 0x01010101u) & ~v & 0x80808080u;
    if (lane == 2) return (v - 0x00010001u) & ~v & 0x80008000u;
    return v == 0u ? 0x80000000u : 0u;
}

// Does any band c < b of x and y agree?  Cosine: packed key rows.
__device__ __forceinline__ bool earlier_band_cos(const BandArgs &A, uint32_t x, uint32_t y, int b) {
    const uint32_t *kx = A.ck + (size_t)x * A.ck_words, *ky = A.ck + (size_t)y * A.ck_words;
    const int per_word = 4 / A.ck_lane;
    const int full = b / per_word, rest = b % per_word;
    for (int w = 0; w < full; ++w)
        if (zero_lanes(__ldg(kx + w) ^ __ldg(ky + w), A.ck_lane)) return true;
    if (rest) {
        const uint32_t keep = (1u << (8 * A.ck_lane * rest)) - 1u;   // the low `rest` lanes
        if (zero_lanes(__ldg(kx + full) ^ __ldg(ky + full), A.ck_lane) & keep) return true;
    }
    return false;
}

// The pair (x, y) met in band b is emitted iff its band-b keys agree in full
// and no earlier band has them agree.
__device__ __forceinline__ bool emit_here(const BandArgs &A, uint32_t x, uint32_t y, int b) {
    if (A.kind == BLSH_COSINE) return !earlier_band_cos(A, x, y, b);
    return emit_here_jaccard(A, x, y, b);
}

// Cosine rows of packed band keys are at most kCkRegWords words long when
// they fit the register fast path below (64 one-byte bands, 32 two-byte
// bands or 16 four-byte bands).
constexpr int kCkRegWords = 16;

// Cosine emission with x's packed keys held in registers: a pair (x, y) of
// band b is checked against bands < b with 16-byte loads of y's key row only.
__device__ __forceinline__ bool earlier_band_cos_reg(const BandArgs &A, const uint4 (&kx)[kCkRegWords / 4],
                                                     uint32_t y, int b) {
    const uint4 *ky = reinterpret_cast<const uint4 *>(A.ck + (size_t)y * A.ck_words);
    const int per_word = 4 / A.ck_lane;
    const int need = (b + per_word - 1) / per_word;   // words holding bands 0..b-1
#pragma unroll
    for (int w4 = 0; w4 < kCkRegWords / 4; ++w4) {
        if (4 * w4 < need) {
            const uint4 yv = __ldg(ky + w4);
            const uint32_t z[4] = {kx[w4].x ^ yv.x, kx[w4].y ^ yv.y, kx[w4].z ^ yv.z, kx[w4].w ^ yv.w};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int w = 4 * w4 + c;
                if (w < need) {
                    const int lanes = (w + 1) * per_word <= b ? per_word : b - w * per_word;
                    const uint32_t keep = lanes == per_word ? 0xffffffffu : (1u << (8 * A.ck_lane * lanes)) - 1u;
                    if (zero_lanes(z[c], A.ck_lane) & keep) return true;
                }
            }
        }
    }
    return false;
}

template <bool WRITE>
__global__ void emit_kernel(BandArgs A, const unsigned long long *keys, const uint32_t *vals, long long n,
                            unsigned long long *counts, uint32_t *pairs, long long cap) {
    // Lanes of a warp take 32 consecutive sorted positions.  A position whose
    // bucket continues for at most 32 more entries walks them alone; longer
    // ones are walked afterwards by the whole warp, 32 partners per step, so
    // a bucket of thousands of objects is not a serial chain of loads.
    const bool reg_path = A.kind == BLSH_COSINE && A.ck_words <= kCkRegWords;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long pb = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); pb < n; pb += stride) {
        const long long p = pb + lane;
        const bool live = p < n;
        unsigned long long key = 0;
        uint32_t x = 0;
        int b = 0;
        bool longrun = false;
        unsigned long long c = 0, out = 0;
        if (live) {
            key = keys[p];
            x = vals[p];
            b = A.kind == BLSH_COSINE ? (int)(key >> A.rows) : (A.band_bits == 0 ? 0 : (int)(key >> A.key_shift));
            out = WRITE ? counts[p] : 0;
            longrun = p + 33 < n && keys[p + 33] == key;
        }
        if (live && !longrun) {
            if (reg_path) {
                uint4 kx[kCkRegWords / 4];
                const uint4 *kxp = reinterpret_cast<const uint4 *>(A.ck + (size_t)x * A.ck_words);
#pragma unroll
                for (int w4 = 0; w4 < kCkRegWords / 4; ++w4)
                    kx[w4] = 4 * w4 < A.ck_words ? __ldg(kxp + w4) : make_uint4(0u, 0u, 0u, 0u);
                for (long long q = p + 1; q < n && keys[q] == key; ++q) {
                    const uint32_t y = vals[q];
                    if (!earlier_band_cos_reg(A, kx, y, b)) {
                        if (WRITE) {
                            const long long o = (long long)(out + c);
                            if (o < cap) reinterpret_cast<uint2 *>(pairs)[o] = make_uint2(x, y);
                        }
                        ++c;
                    }
                }
            } else {
                for (long long q = p + 1; q < n && keys[q] == key; ++q) {
                    const uint32_t y = vals[q];
                    if (emit_here(A, x, y, b)) {
                        if (WRITE) {
                            const long long o = (long long)(out + c);
                            if (o < cap) reinterpret_cast<uint2 *>(pairs)[o] = make_uint2(x, y);
                        }
                        ++c;
                    }
                }
            }
        }
        // the warp walks the long buckets of its lanes, one position at a time
        unsigned pending = __ballot_sync(kFull, longrun);
        while (pending) {
            const int l = __ffs(pending) - 1;
            pending &= pending - 1;
            const long long pl = __shfl_sync(kFull, p, l);
            const unsigned long long kl = __shfl_sync(kFull, key, l);
            const uint32_t xl = __shfl_sync(kFull, x, l);
            const int bl = __shfl_sync(kFull, b, l);
            const unsigned long long ol = __shfl_sync(kFull, out, l);
            unsigned long long cl = 0;
            for (long long q0 = pl + 1;; q0 += 32) {
                const long long q = q0 + lane;
                const bool in = q < n && keys[q] == kl;
                bool ok = false;
                uint32_t y = 0;
                if (in) {
                    y = vals[q];
                    ok = emit_here(A, xl, y, bl);
                }
                const unsigned m = __ballot_sync(kFull, ok);
                if (WRITE && ok) {
                    const long long o = (long long)(ol + cl + __popc(m & lt));
                    if (o < cap) reinterpret_cast<uint2 *>(pairs)[o] = make_uint2(xl, y);
                }
                cl += __popc(m);
                if (__ballot_sync(kFull, in) != kFull) break;   // the bucket ended in this step
            }
            if (lane == l) c = cl;
        }
        if (!WRITE && live) counts[p] = c;
    }
}

// ---- staged emission ----------------------------------------------------------

constexpr int kStageWords = 32;   // key rows of up to 128 bytes take this path
constexpr int kKeyWin = 128;      // keys a warp stages to find its buckets' ends
constexpr unsigned kFewOpen = 48; // open tests per 32 partners up to which rows are not staged whole

// Rows of up to 64 bytes (KW4 = 4 16-byte chunks) and up to 128 (KW4 = 8).
// Per warp: the key rows of its chunk's 32 positions and a few more, kStage of
// them in all, and of a batch of kBatch partners past them.  Staged rows are
// cws = cw4 | 1 16-byte words apart: an odd stride, so that lanes reading
// different rows hit different banks.  The sizes leave room for three CTAs of
// eight warps an SM.
template <int KW4>
struct Emit {
    static constexpr int kStage = KW4 <= 4 ? 64 : 36;
    static constexpr int kBatch = KW4 <= 4 ? 32 : 16;
    static constexpr int kStride = KW4 | 1;   // the largest cws
    // bytes of a warp's region: staged rows, batch rows, keys, ids of the stage,
    // of the batch, undecided tests (KW4 = 8), kept bits
    static constexpr int kRows = kStage * kStride * 16, kBatchRows = kBatch * kStride * 16;
    static constexpr int kList = KW4 <= 4 ? 0 : kBatch * 32 * 2;
    static constexpr int kLite = 96;          // (KW4 = 8) partners whose first chunks alone fit the batch's rows
    static_assert(KW4 <= 4 || kLite * (16 + 4) <= kBatchRows, "first chunks and ids");
    static constexpr int kRegion = kRows + kBatchRows + kKeyWin * 4 + kStage * 4 + 32 * 4 + kList + 32 * 4;
    static_assert(kRegion % 16 == 0, "regions start on 16 bytes");
};

// First position q >= from with q == n or keys[q] != key, given
// keys[from - 1] == key: galloping, then a binary search.
template <typename K>
__device__ long long run_end_global(const K *keys, long long n, long long from, K key) {
    long long lo = from, step = 1;
    while (lo < n && keys[lo] == key) {
        const long long probe = lo + step;
        if (probe >= n || keys[probe] != key) {
            long long hi = probe < n ? probe : n;
            ++lo;
            while (lo < hi) {
                const long long mid = (lo + hi) >> 1;
                if (keys[mid] == key) lo = mid + 1; else hi = mid;
            }
            return lo;
        }
        lo = probe;
        step <<= 1;
    }
    return lo;
}

// Whether any of a set of words has a zero lane of LANE bytes, accumulated over
// 16-byte chunks.  Two- and four-byte lanes keep the smallest lane seen (a
// three-way minimum takes two words an instruction: with the XOR 1.5
// operations a word); bytes have no such instruction and use the borrow test,
// (z - 1) & ~z in every lane, whose false flags lie only above a true one.
template <int LANE>
struct ZeroLanes {
    uint32_t a = LANE == 1 ? 0u : ~0u;
    __device__ __forceinline__ void add(uint32_t z0, uint32_t z1, uint32_t z2, uint32_t z3) {
        if constexpr (LANE == 1) {
            a |= ((z0 - 0x01010101u) & ~z0) | ((z1 - 0x01010101u) & ~z1);
            a |= ((z2 - 0x01010101u) & ~z2) | ((z3 - 0x01010101u) & ~z3);
        } else if constexpr (LANE == 2) {
            a = __vimin3_u16x2(a, z0, z1);
            a = __vimin3_u16x2(a, z2, z3);
        } else {
            a = __vimin3_u32(a, z0, z1);
            a = __vimin3_u32(a, z2, z3);
        }
    }
    __device__ __forceinline__ bool any() const {
        if constexpr (LANE == 1) return (a & 0x80808080u) != 0;
        if constexpr (LANE == 2) return ((a - 0x00010001u) & ~a & 0x80008000u) != 0;
        return a == 0;
    }
};

// Poison for word w of a key row at band b: all ones in every lane of a band
// >= b, zero below; (x ^ y) | poison can be zero only in an earlier band's lane.
template <int LANE>
__device__ __forceinline__ uint32_t poison_word(int w, int b) {
    constexpr int PW = 4 / LANE;   // lanes per word
    const int left = b - w * PW;   // earlier bands in this word
    return left >= PW ? 0u : left <= 0 ? ~0u : ~((1u << (8 * LANE * left)) - 1u);
}

// The tests of one pair of key rows, chunks [K0, nw) of 16 bytes: true when no
// band below b agrees.
template <int K0, int NW4, int LANE, typename XR, typename YR>
__device__ __forceinline__ bool no_earlier_band(const XR &x, const YR &y, int b) {
    constexpr int PC = 16 / LANE;                 // lanes per chunk
    ZeroLanes<LANE> z;
    const int full = b / PC;                      // chunks of earlier bands only
#pragma unroll
    for (int k = K0; k < NW4; ++k) {
        if (k <= full) {
            const uint4 u = x[k], v = y[k];
            uint32_t p0 = 0, p1 = 0, p2 = 0, p3 = 0;
            if (k == full) {
                p0 = poison_word<LANE>(4 * k, b);
                p1 = poison_word<LANE>(4 * k + 1, b);
                p2 = poison_word<LANE>(4 * k + 2, b);
                p3 = poison_word<LANE>(4 * k + 3, b);
            }
            z.add((u.x ^ v.x) | p0, (u.y ^ v.y) | p1, (u.z ^ v.z) | p2, (u.w ^ v.w) | p3);
        }
    }
    return !z.any();
}

// The same for chunks 1 .. b / PC of rows given as pointers, one of them perhaps
// in global memory, with a loop (b is nearly always the same for the whole
// warp: its positions lie in one band).
template <int LANE>
__device__ __forceinline__ bool no_earlier_band_past_first(const uint4 *x, const uint4 *y, int b) {
    const int full = b / (16 / LANE);
    ZeroLanes<LANE> z;
#pragma unroll 2
    for (int k = 1; k < full; ++k) {
        const uint4 u = x[k], v = y[k];
        z.add(u.x ^ v.x, u.y ^ v.y, u.z ^ v.z, u.w ^ v.w);
    }
    if (b % (16 / LANE)) {
        const uint4 u = x[full], v = y[full];
        z.add((u.x ^ v.x) | poison_word<LANE>(4 * full, b), (u.y ^ v.y) | poison_word<LANE>(4 * full + 1, b),
              (u.z ^ v.z) | poison_word<LANE>(4 * full + 2, b), (u.w ^ v.w) | poison_word<LANE>(4 * full + 3, b));
    }
    return !z.any();
}

// Jaccard class ids: whether word b of the two rows agrees (a key collision is
// not a bucket).
__device__ __forceinline__ bool same_class(const uint4 *x, const uint4 *y, int b) {
    return reinterpret_cast<const uint32_t *>(x)[b] == reinterpret_cast<const uint32_t *>(y)[b];
}

// Output of one record word of a walk: lane l's partners with bit t of `bits`
// set (partner ids ids[t], in shared memory) go to positions out, out + 1, ...
// of the list (advanced).  Where few lanes hold most of the bits, their pairs
// are written lane by lane, 32 partners a store; otherwise every lane writes
// its own.
__device__ __forceinline__ void emit_word(uint32_t bits, const uint32_t *ids, uint32_t x, unsigned long long &out,
                                          uint32_t *pairs, long long cap) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    unsigned owners = __ballot_sync(kFull, bits != 0);
    if (!owners) return;
    const int mine = __popc(bits);
    if (__popc(owners) < 3 * (int)__reduce_max_sync(kFull, (unsigned)mine)) {
        const uint32_t y = ids[lane];
        for (; owners; owners &= owners - 1) {
            const int l = __ffs(owners) - 1;
            const uint32_t m = __shfl_sync(kFull, bits, l), xl = __shfl_sync(kFull, x, l);
            const unsigned long long ol = __shfl_sync(kFull, out, l) + __popc(m & lt);
            if (((m >> lane) & 1u) && (long long)ol < cap) reinterpret_cast<uint2 *>(pairs)[ol] = make_uint2(xl, y);
        }
    } else {
        unsigned long long o = out;
        for (uint32_t m = bits; m; m &= m - 1, ++o)
            if ((long long)o < cap) reinterpret_cast<uint2 *>(pairs)[o] = make_uint2(x, ids[__ffs(m) - 1]);
    }
    out += mine;
}

// What the passes keep per position and chunk of positions.
struct EmitState {
    uint32_t *kept;               // [n]: pairs of a position (chunks that walk)
    uint32_t *partners;           // [n]: partners of a position (the rest of its bucket)
    unsigned long long *chunk;    // [chunks]: pairs of a chunk, then their offset
    uint32_t *rec;                // the keep record, rec_cap words
    unsigned long long *rec_off;  // [chunks]: first word * 4 + 2 (split) + 1 (flat), or ~0: not recorded
    unsigned long long rec_cap;
    unsigned long long *next, *rec_next;
    uint2 *tasks;                 // [task_cap]: (chunk, segment) of the split chunks, chunk ~0: unused
    unsigned long long task_cap;
    unsigned long long *task_next;
};

// A chunk whose walk is longer than kSplit partners is cut into segments of kSeg
// partners, tasks of their own for any warp (a bucket of 15,190 of 1e6
// neighbour lists holds 62% of all pairs in 475 chunks: a warp each had left
// seven eighths of the GPU idle for milliseconds).  Its record starts with 32
// words a segment, the pairs each lane keeps there, from which the write pass's
// tasks know their places.
constexpr unsigned kSplit = 2048, kSeg = 1024;
enum EmitMode { kCount, kSegment, kRetest };

// Owner of test t among the warp's positions: the last lane whose exclusive
// prefix `off` is <= t.
__device__ __forceinline__ int owner_of(unsigned t, unsigned off) {
    int o = 0;
#pragma unroll
    for (int step = 16; step > 0; step >>= 1) {
        const unsigned oc = __shfl_sync(kFull, off, o + step);
        if (oc <= t) o += step;
    }
    return o;
}

template <typename T>
__device__ __forceinline__ T warp_exclusive(T v) {
    const int lane = threadIdx.x & 31;
    T incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    return incl - v;
}

// Count pass (kCount, then kSegment for the segments of split chunks) and the
// write pass of the chunks the record had no room for (kRetest).  Warps are
// independent workers: a warp takes the next chunk of 32 sorted positions (or
// segment) from a counter and finds the end of every position's bucket (binary
// search in the staged keys, continued in global memory past them).  Lane l
// owns position l (object x, band b).
//
// Where buckets are long the warp walks the partners of its 32 positions in
// order, kBatch at a time (their key rows loaded 128 contiguous bytes at a
// time, unless they are staged already): each step reads one partner's row, the
// same address for every lane, and every lane tests its own pair on the bands
// before its own.  Rows of more than 64 bytes are first tested on their first
// 16 bytes, which settles nearly every pair that agrees in an earlier band; the
// tests left open are listed in shared memory and dealt one to a lane.  While
// few tests stay open (kFewOpen per 32 partners) only the first 16 bytes of
// the partners' rows are loaded, 96 partners at a time, and an open test reads
// the rest of its partner's row from global memory: in a bucket of thousands
// of near-identical neighbour lists nothing else is needed.  Where
// buckets are short the warp numbers the pairs and gives each lane one
// ("flat").  Pairs come in order of position, then partner.
//
// Keep record: the count pass stores which pairs it keeps, one bit per tested
// pair, so that the write pass only writes them: a chunk takes its words (flat:
// one per 32 pairs; the walk: 32 per 32 partners, word 32 w + l holding
// partners 32 w + 1 .. 32 w + 32 of lane l's chunk) from a counter.
//
// 1e6 points, 64 bands of 16 bits (1.7e9 tests of 6.4e8 pairs): the count
// pass 15.1 ms with borrow tests on every word, whole windows staged a row per
// lane and the open tests dealt by searching their owners; 8.9 now.  Of that
// the open tests take 2.8, the first tests 1.0, loading rows 2 (of a row's
// eight pieces only those that the chunk's bands reach, 4.5 on average; whole
// rows took 0.7 ms more); the pass issues on 6 cycles of 10, two thirds of the
// integer pipe's rate.  (A table of the poison words, more rows staged where
// they are short, and ids at hand for the first batches changed nothing.)
template <int MODE, int KW4, int LANE>
__global__ void __launch_bounds__(256, 3) emit_warp_kernel(BandArgs A, const uint32_t *__restrict__ keys,
                                                           const uint32_t *__restrict__ vals, long long n,
                                                           EmitState E, uint32_t *pairs, long long cap) {
    using R = Emit<KW4>;
    constexpr bool RETEST = MODE == kRetest;
    if (RETEST && (cap == 0 || *E.rec_next <= E.rec_cap)) return;   // nothing to write, or every chunk recorded
    extern __shared__ uint4 s_all[];
    const int cw4 = A.ck_words >> 2, cws = cw4 | 1;
    // 16-byte chunks of a key row that this chunk's bands reach, and i / need = i * magic >> 16 for i < 2^11 (need <= 8)
    int need = cw4;
    unsigned magic = (65536u + cw4 - 1) / cw4;
    const int lane = threadIdx.x & 31;
    unsigned char *region = reinterpret_cast<unsigned char *>(s_all) + (threadIdx.x >> 5) * R::kRegion;
    uint4 *s_ck = reinterpret_cast<uint4 *>(region);
    uint4 *w_rows = reinterpret_cast<uint4 *>(region + R::kRows);
    uint32_t *s_key = reinterpret_cast<uint32_t *>(region + R::kRows + R::kBatchRows);
    uint32_t *s_val = s_key + kKeyWin;
    uint32_t *w_ids = s_val + R::kStage;
    uint32_t *s_und = w_ids + 32;
    [[maybe_unused]] uint16_t *s_list = reinterpret_cast<uint16_t *>(s_und + 32);
    const bool jac = LANE == 4 && A.exact_classes;
    const unsigned long long items =
        MODE == kSegment ? (*E.task_next < E.task_cap ? *E.task_next : E.task_cap) : (unsigned long long)((n + 31) >> 5);
    // the first `need` chunks of the key rows of objects ids[0 .. m) into dst
    auto load_rows = [&](uint4 *dst, const uint32_t *ids, int m) {
#pragma unroll 4
        for (int i = lane; i < m * need; i += 32) {
            const int k = (int)((unsigned)i * magic >> 16), q = i - k * need;
            dst[k * cws + q] = __ldg(reinterpret_cast<const uint4 *>(A.ck + (size_t)ids[k] * A.ck_stride) + q);
        }
    };
    // The next chunk, its keys and its first ids are fetched while this one is
    // worked on: its number, its keys, its ids and its rows would otherwise be
    // four waits one after the other at its start (10.4 ms of the pass below,
    // 9.5 so).  (Every warp starts with the
    // chunk of its own number, so that none holds two while another has none;
    // segments, a few a warp and long, are taken when they are begun.)
    constexpr bool AHEAD = MODE == kCount;
    static_assert(R::kStage <= 64, "two ids a lane");
    uint32_t ahead_key[kKeyWin / 32], ahead_val[2];
    unsigned long long after = 0;                         // (lane 0) the chunk after the next
    const unsigned long long workers = (unsigned long long)gridDim.x * (blockDim.x >> 5);
    auto grab = [&] { after = lane == 0 ? (AHEAD ? workers : 0ull) + atomicAdd(E.next, 1ull) : 0ull; };
    auto fetch = [&](unsigned long long ch) {
        if (!AHEAD || ch >= items) return;
        const long long left = n - (long long)(ch << 5);
#pragma unroll
        for (int q = 0; q < kKeyWin / 32; ++q) ahead_key[q] = lane + 32 * q < left ? __ldg(keys + (ch << 5) + lane + 32 * q) : 0u;
#pragma unroll
        for (int q = 0; q < 2; ++q) ahead_val[q] = lane + 32 * q < left ? __ldg(vals + (ch << 5) + lane + 32 * q) : 0u;
    };
    unsigned long long next = (unsigned long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (AHEAD && next < items) {
        fetch(next);
        grab();
    }
    for (;;) {
        if (!AHEAD) {
            grab();
            next = __shfl_sync(kFull, after, 0);
        }
        unsigned long long c = next;
        if (c >= items) break;
        if (AHEAD) {
            __syncwarp();                                 // the previous chunk is done with the region
#pragma unroll
            for (int q = 0; q < kKeyWin / 32; ++q) s_key[lane + 32 * q] = ahead_key[q];
#pragma unroll
            for (int q = 0; q < 2; ++q)
                if (lane + 32 * q < R::kStage) s_val[lane + 32 * q] = ahead_val[q];
            __syncwarp();
            next = __shfl_sync(kFull, after, 0);
            if (next < items) grab();
            fetch(next);
        }
        if (RETEST && E.rec_off[c] != ~0ull) continue;
        unsigned seg = 0;
        if (MODE == kSegment) {
            const uint2 task = E.tasks[c];
            if (task.x == ~0u) continue;
            c = task.x;
            seg = task.y;
        }
        const long long p0 = (long long)c << 5;
        const int win = (int)(n - p0 < kKeyWin ? n - p0 : kKeyWin);
        const int tile = win < 32 ? win : 32;
        const bool live = lane < tile;
        // this position's band, and its bucket's end (relative to p0)
        const int b = live ? (int)((uint32_t)(p0 + lane) / (uint32_t)A.N) : 0;
        unsigned end = (unsigned)lane + 1;
        __syncwarp();                                     // the previous chunk is done with the region
        if (MODE == kSegment) {
            if (live) end += E.partners[p0 + lane];
        } else {
            if (!AHEAD) {
                for (int k = lane; k < win; k += 32) s_key[k] = __ldg(keys + p0 + k);
                __syncwarp();
            }
            if (live) {
                const long long band_end = (long long)(b + 1) * A.N - p0;
                const uint32_t key = s_key[lane];
                int lo = lane + 1, hi = band_end < win ? (int)band_end : win;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (s_key[mid] == key) lo = mid + 1; else hi = mid;
                }
                end = (unsigned)lo;
                if (lo == win && band_end > win)
                    end = (unsigned)(run_end_global<uint32_t>(keys, p0 + band_end, p0 + lo, key) - p0);
            }
        }
        const unsigned mine = live ? end - lane - 1 : 0u;   // partners
        const unsigned jmax = __reduce_max_sync(kFull, live ? end : 0u);   // partners are positions 1 .. jmax - 1
        const unsigned pairs_w = __reduce_add_sync(kFull, mine);
        const int staged = (int)(jmax < (unsigned)R::kStage ? jmax : (unsigned)R::kStage);
        if (MODE == kCount && live) E.partners[p0 + lane] = mine;
        if (jmax <= 1 || !__any_sync(kFull, mine != 0)) {
            if (MODE == kCount && lane == 0) {
                E.chunk[c] = 0;
                E.rec_off[c] = 1ull;                      // flat, no words
            }
            continue;
        }
        if (!AHEAD) {
            for (int k = lane; k < staged; k += 32) s_val[k] = __ldg(vals + p0 + k);
            __syncwarp();
        }
        const bool flat = MODE != kSegment && jmax <= (unsigned)R::kStage && 5u * ((pairs_w + 31) / 32) < 2u * (jmax - 1);
        const unsigned segs = MODE == kCount && jmax - 1 > kSplit ? (jmax - 2) / kSeg + 1 : 0u;
        const unsigned long long words = flat ? (pairs_w + 31) / 32 : 32ull * ((jmax + 30) / 32) + 32ull * segs;
        unsigned long long off = 0;                       // (the answer is waited for after the rows)
        if (MODE == kCount && lane == 0) off = atomicAdd(E.rec_next, words);
        // chunks of 16 bytes that any lane's earlier bands (and its class id) reach
        const int nw4 = (int)(__reduce_max_sync(kFull, live ? (unsigned)(b * LANE + 15) / 16 : 0u));
        const int reach = jac ? (int)__reduce_max_sync(kFull, (unsigned)b) / 4 + 1 : nw4 > 0 ? nw4 : 1;
        if (reach != need) {
            need = reach;
            magic = (65536u + reach - 1) / reach;
        }
        load_rows(s_ck, s_val, staged);
        __syncwarp();
        const uint32_t x = live ? s_val[lane] : 0u;
        uint32_t *crec = nullptr;
        unsigned long long out = RETEST ? E.chunk[c] : 0ull;
        if (MODE == kCount) {
            unsigned long long slot = 0;
            if (lane == 0 && segs && off + words <= E.rec_cap) slot = atomicAdd(E.task_next, (unsigned long long)segs);
            off = __shfl_sync(kFull, off, 0);
            slot = __shfl_sync(kFull, slot, 0);
            const bool room = off + words <= E.rec_cap;
            const bool split = segs && room && slot + segs <= E.task_cap;
            if (lane == 0) E.rec_off[c] = room ? off << 2 | (split ? 2ull : 0ull) | (flat ? 1ull : 0ull) : ~0ull;
            if (segs && room)   // its tasks, or (no room for all) slots left unused
                for (unsigned i = lane; i < segs; i += 32)
                    if (slot + i < E.task_cap) E.tasks[slot + i] = make_uint2(split ? (uint32_t)c : ~0u, i);
            if (split) {
                if (live) E.kept[p0 + lane] = 0;
                if (lane == 0) E.chunk[c] = 0;
                continue;
            }
            if (room) crec = E.rec + off;
        } else if (MODE == kSegment) {
            crec = E.rec + (E.rec_off[c] >> 2) + 32ull * ((jmax - 2) / kSeg + 1);
        }
        if (flat) {
            const unsigned off = warp_exclusive(mine);
            unsigned total = 0;
            for (unsigned t0 = 0; t0 < pairs_w; t0 += 32) {
                const unsigned t = t0 + lane;
                const int o = owner_of(t, off);
                const int bo = __shfl_sync(kFull, b, o);
                const int j = o + 1 + (int)(t - __shfl_sync(kFull, off, o));
                bool ok = false;
                if (t < pairs_w) {
                    const uint4 *xr = s_ck + o * cws, *yr = s_ck + j * cws;
                    ok = no_earlier_band<0, KW4, LANE>(xr, yr, bo) && (!jac || same_class(xr, yr, bo));
                }
                const unsigned okm = __ballot_sync(kFull, ok);
                if (MODE == kCount && crec && lane == 0) crec[t0 >> 5] = okm;
                if (RETEST && ok) {
                    const long long slot = (long long)out + __popc(okm & ((1u << lane) - 1u));
                    if (slot < cap) reinterpret_cast<uint2 *>(pairs)[slot] = make_uint2(s_val[o], s_val[j]);
                }
                if (RETEST) out += __popc(okm);
                total += __popc(okm);
            }
            if (MODE == kCount && lane == 0) E.chunk[c] = total;
            continue;
        }
        if (RETEST) {   // each lane's first output
            const unsigned long long kept = live ? E.kept[p0 + lane] : 0u;
            out += warp_exclusive(kept);
        }
        // the walk; a lane's poison for its first chunks, its partners lane < j < end
        constexpr int PZ = KW4 <= 4 ? 4 * KW4 : 4;
        uint32_t pz[PZ];
        uint4 kx[PZ / 4];
#pragma unroll
        for (int w = 0; w < PZ; ++w) pz[w] = poison_word<LANE>(w, b);
#pragma unroll
        for (int k = 0; k < PZ / 4; ++k) kx[k] = live && k < cw4 ? s_ck[lane * cws + k] : make_uint4(0u, 0u, 0u, 0u);
        const uint32_t xb = jac ? reinterpret_cast<const uint32_t *>(s_ck + (live ? lane : 0) * cws)[b] : 0u;
        // (KW4 = 8) tests past the first chunk: earlier bands, or a class id, there
        const bool more = b * LANE > 16 || (jac && b >= 4);
        unsigned cnt = 0;
        uint32_t racc = 0;
        // partners j0 .. j0 + m - 1 against the first PZ / 4 chunks (rows
        // `stride` chunks apart): bit u set where none of their earlier bands
        // agrees (and band b's class does, if it lies in the chunks read)
        auto batch = [&](auto nchunks, const uint4 *rows, int stride, int m, bool with_class) {
            constexpr int NC = decltype(nchunks)::value;
            uint32_t keep = 0;
            for (int u0 = 0; u0 < m; u0 += 8) {           // (rows past m are read, inside the region, and masked)
                uint32_t k8 = 0;
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const uint4 *row = rows + (u0 + u) * stride;
                    ZeroLanes<LANE> z;
#pragma unroll
                    for (int k = 0; k < NC; ++k) {
                        const uint4 v = row[k];
                        z.add((kx[k].x ^ v.x) | pz[4 * k], (kx[k].y ^ v.y) | pz[4 * k + 1],
                              (kx[k].z ^ v.z) | pz[4 * k + 2], (kx[k].w ^ v.w) | pz[4 * k + 3]);
                    }
                    bool ok = !z.any();
                    if (LANE == 4 && with_class) ok = ok && reinterpret_cast<const uint32_t *>(row)[b] == xb;
                    if (ok) k8 |= 1u << u;
                }
                keep |= k8 << u0;
            }
            return keep;
        };
        // this lane's partners among j0 .. j0 + m - 1 (m <= 32): lane < j0 + u < end
        auto range_of = [&](unsigned j0, int m) {
            const unsigned lo = (unsigned)lane + 1 > j0 ? ((unsigned)lane + 1 - j0 < 32u ? lane + 1 - j0 : 32u) : 0u;
            const unsigned hi = live && end > j0 ? (end - j0 < (unsigned)m ? end - j0 : (unsigned)m) : 0u;
            return (hi >= 32u ? ~0u : (1u << hi) - 1u) & ~(lo >= 32u ? ~0u : (1u << lo) - 1u);
        };
        // (KW4 = 8) the tests of `open`, dealt one to a lane: partner u's row
        // is rows + u cws, or (ids given) in global memory; returns the bits
        // that stay
        auto deal = [&](uint32_t open, unsigned total, const uint4 *rows, const uint32_t *ids) {
            unsigned off = warp_exclusive((unsigned)__popc(open));
            __syncwarp();
            s_und[lane] = 0;
            for (uint32_t m2 = open; m2; m2 &= m2 - 1) s_list[off++] = (uint16_t)(lane << 5 | (__ffs(m2) - 1));
            __syncwarp();
            for (unsigned t0 = 0; t0 < total; t0 += 32) {
                const bool have = t0 + lane < total;
                const unsigned e = have ? s_list[t0 + lane] : 0u;
                const int o = (int)(e >> 5), u = (int)(e & 31);
                const int bo = __shfl_sync(kFull, b, o);
                if (have) {
                    const uint4 *xr = s_ck + o * cws;
                    const uint4 *yr = ids ? reinterpret_cast<const uint4 *>(A.ck + (size_t)ids[u] * A.ck_stride)
                                          : rows + u * cws;
                    if (no_earlier_band_past_first<LANE>(xr, yr, bo) && (!jac || same_class(xr, yr, bo)))
                        atomicOr(&s_und[o], 1u << u);
                }
            }
            __syncwarp();
            return s_und[lane];
        };
        // a finished record word: partners 32 w + 1 .. 32 w + 32
        auto put_word = [&](unsigned w, uint32_t word, const uint32_t *ids) {
            cnt += __popc(word);
            if (!RETEST && crec) crec[(size_t)w * 32 + lane] = word;
            if (RETEST) {
                __syncwarp();
                emit_word(word, ids, x, out, pairs, cap);
                __syncwarp();
            }
        };
        [[maybe_unused]] unsigned open_word = 0;          // tests the last word left open after its first chunk
        const unsigned first = 1 + (MODE == kSegment ? seg * kSeg : 0u);
        const unsigned jend = MODE == kSegment && jmax - first > kSeg ? first + kSeg : jmax;
        for (unsigned j0 = first; j0 < jend;) {
            if constexpr (KW4 > 4) {
                if (((j0 - 1) & 31) == 0 && (int)j0 >= staged && open_word <= kFewOpen) {
                    // first chunks only, R::kLite partners
                    uint4 *rows0 = w_rows;
                    uint32_t *ids = reinterpret_cast<uint32_t *>(rows0 + R::kLite);
                    __syncwarp();
#pragma unroll
                    for (int q = 0; q < R::kLite / 32; ++q) {
                        const unsigned j = j0 + 32 * q + lane;
                        if (j < jend) ids[32 * q + lane] = __ldg(vals + p0 + j);
                    }
#pragma unroll
                    for (int q = 0; q < R::kLite / 32; ++q) {
                        const unsigned j = j0 + 32 * q + lane;
                        if (j < jend)
                            rows0[32 * q + lane] =
                                __ldg(reinterpret_cast<const uint4 *>(A.ck + (size_t)ids[32 * q + lane] * A.ck_stride));
                    }
                    __syncwarp();
                    open_word = 0;
                    for (int q = 0; q < R::kLite / 32 && j0 < jend; ++q, j0 += 32) {
                        const int m = (int)(jend - j0 < 32u ? jend - j0 : 32u);
                        uint32_t keep = batch(std::integral_constant<int, 1>{}, rows0 + 32 * q, 1, m, jac && b < 4) &
                                        range_of(j0, m);
                        const uint32_t open = more ? keep : 0u;
                        const unsigned total = __reduce_add_sync(kFull, (unsigned)__popc(open));
                        if (total) {   // (the list holds the tests of 16 partners)
                            uint32_t stay = 0;
#pragma unroll 1
                            for (int hf = 0; hf < 2; ++hf) {
                                const uint32_t part = open & (hf ? 0xffff0000u : 0xffffu);
                                const unsigned np = __reduce_add_sync(kFull, (unsigned)__popc(part));
                                if (np) stay |= deal(part, np, nullptr, ids + 32 * q);
                            }
                            if (more) keep = stay;
                        }
                        open_word = total > open_word ? total : open_word;
                        put_word((j0 - 1) >> 5, keep, ids + 32 * q);
                    }
                    continue;
                }
            }
            const int m = (int)(jend - j0 < (unsigned)R::kBatch ? jend - j0 : (unsigned)R::kBatch);
            const unsigned at = (j0 - 1) & 31;            // a record word holds 32 partners: one batch or two
            const uint4 *rows = s_ck + j0 * cws;
            const bool inside = (int)j0 + m <= staged;
            if (!inside || RETEST) {
                __syncwarp();
                if (lane < m) w_ids[at + lane] = __ldg(vals + p0 + j0 + lane);
                __syncwarp();
            }
            if (!inside) {
                load_rows(w_rows, w_ids + at, m);
                __syncwarp();
                rows = w_rows;
            }
            const uint32_t range = range_of(j0, m);
            uint32_t keep = 0;
            if (!__any_sync(kFull, range != 0)) {
                // no lane has a partner here (buckets end and begin inside the chunk)
            } else if constexpr (KW4 <= 4) {
                switch (nw4) {
                case 0: keep = batch(std::integral_constant<int, 0>{}, rows, cws, m, jac); break;
                case 1: keep = batch(std::integral_constant<int, 1>{}, rows, cws, m, jac); break;
                case 2: keep = batch(std::integral_constant<int, 2>{}, rows, cws, m, jac); break;
                case 3: keep = batch(std::integral_constant<int, 3>{}, rows, cws, m, jac); break;
                default: keep = batch(std::integral_constant<int, 4>{}, rows, cws, m, jac); break;
                }
                keep &= range;
            } else {
                // the first chunk; lanes with earlier bands past it have open tests left
                keep = batch(std::integral_constant<int, 1>{}, rows, cws, m, jac && b < 4) & range;
                const uint32_t open = more ? keep : 0u;
                const unsigned total = __reduce_add_sync(kFull, (unsigned)__popc(open));
                if (total) {
                    const uint32_t stay = deal(open, total, rows, nullptr);
                    if (more) keep = stay;
                }
                open_word = at == 0 ? total : open_word + total;
            }
            racc = at == 0 ? keep : racc | keep << at;
            if (at + R::kBatch == 32 || j0 + R::kBatch >= jend) put_word((j0 - 1) >> 5, racc, w_ids);
            j0 += R::kBatch;
        }
        if (!RETEST) {
            const unsigned long long total = (unsigned long long)__reduce_add_sync(kFull, cnt & 0xffffu) +
                                             ((unsigned long long)__reduce_add_sync(kFull, cnt >> 16) << 16);
            if (MODE == kSegment) {
                E.rec[(E.rec_off[c] >> 2) + 32ull * seg + lane] = cnt;
                if (live && cnt) atomicAdd(E.kept + p0 + lane, cnt);
                if (lane == 0 && total) atomicAdd(E.chunk + c, total);
            } else {
                if (live) E.kept[p0 + lane] = cnt;
                if (lane == 0) E.chunk[c] = total;
            }
        }
    }
}

// The write pass of the recorded chunks: no key or key row is read.  Where a
// chunk's pairs fit the warp's stage (kOutStage of them) they are put in order
// in shared memory first, so that they leave in coalesced stores: the positions
// of a chunk hold consecutive runs of the list.
// 6.4e8 pairs of 64 bands: 7.1 ms with every lane storing its own pairs,
// 2.6 now; 1e9 pairs of 5 bands 4.7 ms, 2.4 now.
// SEG: the segments of split chunks instead.
constexpr int kOutStage = 704;
template <bool SEG>
__global__ void __launch_bounds__(256) emit_write_kernel(const uint32_t *__restrict__ vals, long long n, EmitState E,
                                                         uint32_t *pairs, long long cap,
                                                         const long long *n_pairs, blsh_dev_scratch *scratch) {
    __shared__ __align__(16) uint2 s_out[8][kOutStage];
    __shared__ uint32_t s_ids[8][64];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    uint2 *stage = s_out[warp];
    uint32_t *ids = s_ids[warp];
    if (!SEG && blockIdx.x == 0 && threadIdx.x == 0 && *n_pairs > cap)
        blsh_dev_error(scratch, BLSH_ETRUNC, 1, (unsigned long long)(*n_pairs - cap));
    if (cap == 0) return;                                 // a count-only call
    const long long chunks = (n + 31) >> 5;
    const unsigned long long items =
        SEG ? (*E.task_next < E.task_cap ? *E.task_next : E.task_cap) : (unsigned long long)chunks;
    for (;;) {
        unsigned long long c = 0;
        if (lane == 0) c = atomicAdd(E.next, 1ull);
        c = __shfl_sync(kFull, c, 0);
        if (c >= items) break;
        unsigned seg = 0;
        if (SEG) {
            const uint2 task = E.tasks[c];
            if (task.x == ~0u) continue;
            c = task.x;
            seg = task.y;
        }
        const unsigned long long ro = E.rec_off[c];
        // not recorded: tested again by emit_warp_kernel; split: its segments
        if (ro == ~0ull || (!SEG && (ro & 2ull))) continue;
        const unsigned long long base = E.chunk[c];
        const unsigned long long after = (long long)c + 1 < chunks ? E.chunk[c + 1] : (unsigned long long)*n_pairs;
        const unsigned total = after - base < 0xffffffffull ? (unsigned)(after - base) : 0xffffffffu;
        if (total == 0) continue;
        const uint32_t *rec = E.rec + (ro >> 2);
        const long long p0 = (long long)c << 5;
        const bool live = p0 + lane < n;
        const unsigned mine = live ? E.partners[p0 + lane] : 0u;
        __syncwarp();                                     // the previous chunk's stage has been written out
        if (!SEG && (ro & 1ull)) {   // flat: pairs numbered by position, then partner
            const unsigned pairs_w = __reduce_add_sync(kFull, mine);
            for (int k = lane; k < 64; k += 32) ids[k] = p0 + k < n ? __ldg(vals + p0 + k) : 0u;   // all its partners
            const unsigned off = warp_exclusive(mine);
            __syncwarp();
            unsigned long long o0 = base;
            for (unsigned t0 = 0; t0 < pairs_w; t0 += 32) {
                const unsigned okm = __ldg(rec + (t0 >> 5));
                if (okm) {
                    const unsigned t = t0 + lane;
                    const int o = owner_of(t, off);
                    const int j = o + 1 + (int)(t - __shfl_sync(kFull, off, o));
                    const long long slot = (long long)(o0 + __popc(okm & lt));
                    if (((okm >> lane) & 1u) && slot < cap)
                        reinterpret_cast<uint2 *>(pairs)[slot] = make_uint2(ids[o], ids[j]);
                    o0 += __popc(okm);
                }
            }
            continue;
        }
        const uint32_t x = live ? __ldg(vals + p0 + lane) : 0u;
        const unsigned kept = live ? E.kept[p0 + lane] : 0u;
        const unsigned jmax = __reduce_max_sync(kFull, live ? mine + lane + 1 : 0u);
        unsigned words = (jmax + 30) / 32, w0 = 0;
        if (SEG) {
            w0 = seg * (kSeg / 32);
            words = words - w0 < kSeg / 32 ? words : w0 + kSeg / 32;
        }
        if (!SEG && total <= kOutStage) {
            unsigned o = warp_exclusive(kept);
            for (unsigned w = 0; w < words; ++w) {
                uint32_t bits = __ldg(rec + (size_t)w * 32 + lane);
                const long long q = p0 + 1 + 32ll * w + lane;
                __syncwarp();
                ids[lane] = q < n ? __ldg(vals + q) : 0u;
                __syncwarp();
                for (; bits; bits &= bits - 1) stage[o++] = make_uint2(x, ids[__ffs(bits) - 1]);
            }
            __syncwarp();
            for (unsigned i = lane; i < total; i += 32)
                if ((long long)(base + i) < cap) reinterpret_cast<uint2 *>(pairs)[base + i] = stage[i];
        } else {
            unsigned long long out = base + warp_exclusive<unsigned long long>(kept);
            if (SEG) {   // past the earlier segments' pairs of this lane, and the header
                for (unsigned q = 0; q < seg; ++q) out += __ldg(rec + 32ull * q + lane);
                rec += 32ull * ((jmax - 2) / kSeg + 1);
            }
            for (unsigned w = w0; w < words; ++w) {
                const uint32_t bits = __ldg(rec + (size_t)w * 32 + lane);
                const long long q = p0 + 1 + 32ll * w + lane;
                __syncwarp();
                ids[lane] = q < n ? __ldg(vals + q) : 0u;
                __syncwarp();
                emit_word(bits, ids, x, out, pairs, cap);
            }
        }
    }
}

// ---- staged keys ---------------------------------------------------------------

// The 32-bit key of a band, without the band index: the sign bits themselves,
// or the top 32 - band_bits bits of the band's hash (equal keys are sorted
// together; the class ids split collisions).  row: in shared or global memory.
__device__ __forceinline__ uint32_t band_key32(const BandArgs &A, const uint32_t *row, int b) {
    if (A.kind == BLSH_COSINE) {
        const int start = b * A.rows, w = start >> 5, o = start & 31;
        unsigned long long two = row[w];
        if (o + A.rows > 32) two |= (unsigned long long)row[w + 1] << 32;
        return (uint32_t)(two >> o) & (A.rows == 32 ? ~0u : (1u << A.rows) - 1u);
    }
    unsigned long long h = 0x243f6a8885a308d3ull;
    for (int r = 0; r < A.rows; ++r) h = mix64(h ^ (row[b * A.rows + r] + 0x9e3779b97f4a7c15ull * (r + 1)));
    return (uint32_t)(h >> (32 + A.band_bits));
}

// Word w of a cosine key row packed from its bands' bits.
__device__ __forceinline__ uint32_t packed_word(const BandArgs &A, const uint32_t *row, int w) {
    const int per_word = 4 / A.ck_lane;
    uint32_t v = 0;
    for (int l = 0; l < per_word; ++l) {
        const int b = w * per_word + l;
        if (b < A.bands) v |= band_key32(A, row, b) << (8 * A.ck_lane * l);
    }
    return v;
}

// Keys of every (band, object), bands one after the other, from tiles of
// `objs` signature rows staged in shared memory: the rows are read once, in
// order, and every band's keys leave in runs of objs.  (One thread per (band,
// object) read a 32-byte sector for every key and stored the packed rows two
// bytes at a time: 1.98 ms at 1e6 x 64 bands of 16 bits, 0.16 here.)
// pack: also the cosine key rows (where the signature rows are not they).
// words = 0: rows too long to stage, read from global memory.
__global__ void __launch_bounds__(256) band_keys32_kernel(BandArgs A, uint32_t *__restrict__ keys,
                                                          uint32_t *__restrict__ ck, int words, int objs, bool pack) {
    extern __shared__ uint32_t s_rows[];
    const int stride = words ? words | 1 : A.W;
    const int oshift = 31 - __clz(objs);                  // objs is a power of two
    const long long tiles = (A.N + objs - 1) >> oshift;
    for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
        const long long i0 = t << oshift;
        const int m = (int)(A.N - i0 < objs ? A.N - i0 : objs);
        const uint32_t *rows = words ? s_rows : A.sig + (size_t)i0 * A.W;
        __syncthreads();
        for (int r = threadIdx.x >> 5; r < m; r += 8)
            for (int w = threadIdx.x & 31; w < words; w += 32)
                s_rows[r * stride + w] = __ldg(A.sig + (size_t)(i0 + r) * A.W + w);
        __syncthreads();
        for (int e = threadIdx.x; e < A.bands << oshift; e += 256) {
            const int b = e >> oshift, i = e & (objs - 1);
            if (i < m) keys[(size_t)b * A.N + i0 + i] = band_key32(A, rows + (size_t)i * stride, b);
        }
        if (pack)
            for (int e = threadIdx.x; e < m * A.ck_words; e += 256) {
                const int i = e / A.ck_words, w = e - i * A.ck_words;
                ck[(size_t)(i0 + i) * A.ck_words + w] = packed_word(A, rows + (size_t)i * stride, w);
            }
    }
}

// Jaccard class ids: for sorted position p (object v, band b) the id is the
// first position of its run whose band-b hashes equal v's, so two objects
// share an id in band b iff they agree on the whole band.  Almost always
// that is the run's first position; a hash collision inside a run is split
// off by comparing the hashes themselves.
__global__ void __launch_bounds__(256) class_id_kernel(BandArgs A, uint32_t *ck, const uint32_t *keys,
                                                       const uint32_t *vals, long long n) {
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < n;
         p += (long long)gridDim.x * blockDim.x) {
        const uint32_t key = keys[p];
        const uint32_t v = vals[p];
        const int b = (int)((uint32_t)p / (uint32_t)A.N);
        const long long first = (long long)b * A.N;       // the band's positions start here
        long long cid = p;
        if (p > first && keys[p - 1] == key) {
            // the run's first position: galloping backwards, then a binary search
            long long hi = p, lo = first, step = 1;
            for (;;) {
                const long long probe = hi - step;
                if (probe < first) break;
                if (keys[probe] != key) {
                    lo = probe + 1;
                    break;
                }
                hi = probe;
                step <<= 1;
            }
            while (lo < hi) {
                const long long mid = (lo + hi) >> 1;
                if (keys[mid] == key) hi = mid; else lo = mid + 1;
            }
            if (same_band(A, v, vals[lo], b)) {
                cid = lo;
            } else {
                for (long long q = lo + 1; q < p; ++q)
                    if (same_band(A, v, vals[q], b)) { cid = q; break; }
            }
        }
        ck[(size_t)v * A.ck_words + b] = (uint32_t)cid;
    }
}

// Small object sets: one CTA per band forms the band's keys, sorts them in
// shared memory (the ranking of radix.cuh, eight bits a digit) and writes keys
// and objects in order, with the class ids (Jaccard) or the packed key rows.
// One launch of about 20 us for the 24 of the tiled sort, which at these sizes
// are all latency: 2,000 objects, 32 bands 205 us, 29 here.
constexpr int kSmallObjs = 4096;
constexpr int kSmallWarps = 16;
__global__ void __launch_bounds__(32 * kSmallWarps) band_small_kernel(BandArgs A, int key_bits,
                                                                      uint32_t *__restrict__ keys,
                                                                      uint32_t *__restrict__ vals,
                                                                      uint32_t *__restrict__ ck, bool pack) {
    constexpr int T = 32 * kSmallWarps, ROUNDS = kSmallObjs / T;
    __shared__ uint32_t s_key[kSmallObjs];
    __shared__ uint16_t s_obj[kSmallObjs];
    __shared__ uint32_t cnt[kSmallWarps][256];
    __shared__ uint32_t s_start[256];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, b = blockIdx.x;
    const int N = (int)A.N;
    const int rounds = (N + T - 1) / T;                   // items a lane holds
    const int base = w * rounds * 32 + lane;              // warp w: items [w rounds 32, (w + 1) rounds 32)
    uint32_t key[ROUNDS], rank[ROUNDS];
    uint16_t obj[ROUNDS];
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        const int i = base + 32 * r;
        key[r] = 0;
        obj[r] = (uint16_t)i;
        if (r < rounds && i < N) key[r] = band_key32(A, A.sig + (size_t)i * A.W, b);
    }
    for (int bit = 0; bit < key_bits; bit += 8) {
        for (int d = lane; d < 256; d += 32) cnt[w][d] = 0;
        __syncwarp();
        blsh_radix::warp_ranks<8, ROUNDS>(cnt[w], rank, [&](int r, bool &ok) {
            ok = r < rounds && base + 32 * r < N;
            return (key[r] >> bit) & 255u;
        });
        __syncthreads();
        uint32_t total = 0;
        if (threadIdx.x < 256)
            for (int ww = 0; ww < kSmallWarps; ++ww) {
                const uint32_t c = cnt[ww][threadIdx.x];
                cnt[ww][threadIdx.x] = total;
                total += c;
            }
        const uint32_t start = blsh_scan::block_exclusive<uint32_t>(total, nullptr);
        if (threadIdx.x < 256) s_start[threadIdx.x] = start;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < ROUNDS; ++r)
            if (r < rounds && base + 32 * r < N) {
                const uint32_t d = (key[r] >> bit) & 255u;
                const uint32_t pos = s_start[d] + cnt[w][d] + rank[r];
                s_key[pos] = key[r];
                s_obj[pos] = obj[r];
            }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < ROUNDS; ++r)
            if (r < rounds && base + 32 * r < N) {
                key[r] = s_key[base + 32 * r];
                obj[r] = s_obj[base + 32 * r];
            }
    }
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        const int p = base + 32 * r;
        if (r >= rounds || p >= N) continue;
        keys[(size_t)b * N + p] = key[r];
        vals[(size_t)b * N + p] = obj[r];
        if (A.exact_classes) {
            int cid = p;
            if (p > 0 && s_key[p - 1] == key[r]) {
                int lo = 0, hi = p;                       // the run's first position
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (s_key[mid] < key[r]) lo = mid + 1; else hi = mid;
                }
                if (same_band(A, obj[r], s_obj[lo], b)) {
                    cid = lo;
                } else {
                    for (int q = lo + 1; q < p; ++q)
                        if (same_band(A, obj[r], s_obj[q], b)) { cid = q; break; }
                }
            }
            ck[(size_t)obj[r] * A.ck_words + b] = (uint32_t)(b * N + cid);
        }
    }
    if (pack)   // the bands share the objects' rows out among their CTAs
        for (long long e = (long long)b * T + threadIdx.x; e < (long long)N * A.ck_words; e += (long long)gridDim.x * T) {
            const int i = (int)(e / A.ck_words), wd = (int)(e - (long long)i * A.ck_words);
            ck[e] = packed_word(A, A.sig + (size_t)i * A.W, wd);
        }
}

__global__ void check_cap_kernel(const long long *n_pairs, long long cap, blsh_dev_scratch *scratch) {
    if (*n_pairs > cap) blsh_dev_error(scratch, BLSH_ETRUNC, 1, (unsigned long long)(*n_pairs - cap));
}

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

struct Layout {
    size_t keys0, keys1, vals0, vals1, bk, ck, counts, hist, partial, grand, rec_off, rec, total;
};

// The emission's keep record (emit_warp_kernel): 16 words per position by
// default; bytes a caller's workspace has beyond rec go to it.
constexpr size_t kRecBytesPerPos = 64;

// Jaccard class-id rows: one 32-bit id per band, rounded to 16 bytes.
int jac_row_words(int bands) { return (bands + 3) & ~3; }

Layout layout(long long N, int kind, int rows, int bands) {
    const long long n = N * bands;
    const long long tiles = (n + kSortTile - 1) / kSortTile;
    const long long hist_n = 256 * tiles;
    const long long part = blsh_scan::tiles_for(hist_n > n ? hist_n : n) + 1;
    Layout L;
    size_t o = 0;
    L.keys0 = o; o = up256(o + n * 8);
    L.keys1 = o; o = up256(o + n * 8);
    L.vals0 = o; o = up256(o + n * 4);
    L.vals1 = o; o = up256(o + n * 4);
    const bool classes = kind == BLSH_JACCARD && jac_row_words(bands) <= kStageWords;
    L.bk = o; o = up256(o + (kind == BLSH_JACCARD && !classes ? n * 8 : 0));
    L.ck = o; o = up256(o + (kind == BLSH_COSINE ? (size_t)N * cos_row_words(rows, bands) * 4
                                                  : (classes ? (size_t)N * jac_row_words(bands) * 4 : 0)));
    L.counts = o; o = up256(o + n * 8);
    L.hist = o; o = up256(o + hist_n * 4);
    L.partial = o; o = up256(o + part * 8);
    L.grand = o; o = up256(o + 16);
    L.rec_off = o; o = up256(o + ((n + 31) / 32) * 8);
    L.rec = o;
    L.total = o + (size_t)n * kRecBytesPerPos;
    return L;
}

int band_bits_for(int bands) {
    int b = 0;
    while ((1 << b) < bands) ++b;
    return b;
}

}  // namespace

namespace {

template <int MODE, int KW4, int LANE>
int emit_launch(blsh_ctx *ctx, const BandArgs &A, const uint32_t *keys, const uint32_t *vals, long long n,
                const EmitState &E, uint32_t *pairs, long long cap, cudaStream_t s) {
    constexpr int smem = 8 * Emit<KW4>::kRegion;
    BLSH_CUDA(ctx, cudaFuncSetAttribute(emit_warp_kernel<MODE, KW4, LANE>,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    const long long blocks = (n + 255) / 256, most = (long long)ctx->sm_count * 3;   // a chunk of 32 positions a warp
    blsh_time_start(ctx, s);
    emit_warp_kernel<MODE, KW4, LANE><<<(unsigned)(blocks < most ? blocks : most), 256, smem, s>>>(A, keys, vals, n, E,
                                                                                                    pairs, cap);
    BLSH_LAUNCHED(ctx, MODE == kRetest    ? "emit_warp_kernel (unrecorded chunks)"
                       : MODE == kSegment ? "emit_warp_kernel (count pass, segments)"
                                          : "emit_warp_kernel (count pass)");
    return BLSH_OK;
}

template <int MODE>
int emit_dispatch(blsh_ctx *ctx, const BandArgs &A, const uint32_t *keys, const uint32_t *vals, long long n,
                  const EmitState &E, uint32_t *pairs, long long cap, cudaStream_t s) {
    const bool narrow = A.ck_words <= 16;
    switch (A.ck_lane) {
    case 1: return narrow ? emit_launch<MODE, 4, 1>(ctx, A, keys, vals, n, E, pairs, cap, s)
                          : emit_launch<MODE, 8, 1>(ctx, A, keys, vals, n, E, pairs, cap, s);
    case 2: return narrow ? emit_launch<MODE, 4, 2>(ctx, A, keys, vals, n, E, pairs, cap, s)
                          : emit_launch<MODE, 8, 2>(ctx, A, keys, vals, n, E, pairs, cap, s);
    default: return narrow ? emit_launch<MODE, 4, 4>(ctx, A, keys, vals, n, E, pairs, cap, s)
                           : emit_launch<MODE, 8, 4>(ctx, A, keys, vals, n, E, pairs, cap, s);
    }
}

// Keys of 32 bits sorted band by band, then the staged emission.  The 32-bit
// arrays live in the workspace's regions for 64-bit ones: keys and per-position
// numbers take the lower halves of keys0 and keys1, the sort's histograms (at
// most 2 KB per 4,096 objects and band, and N > 4,096: below 2 n bytes) and the
// partner counts the upper ones.
int staged_candidates(blsh_ctx *ctx, BandArgs &A, const Layout &L, char *ws, size_t workspace_bytes, uint32_t *pairs,
                      int64_t cap, int64_t *n_pairs, cudaStream_t s) {
    const long long N = A.N, n = N * A.bands;
    uint32_t *keys[2] = {(uint32_t *)(ws + L.keys0), (uint32_t *)(ws + L.keys1)};
    uint32_t *vals[2] = {(uint32_t *)(ws + L.vals0), (uint32_t *)(ws + L.vals1)};
    const int key_bits = A.kind == BLSH_COSINE ? A.rows : 32 - A.band_bits;
    // cosine: the signature row is the key row where its lanes are the bands
    bool pack = false;
    if (A.kind == BLSH_COSINE) {
        if (A.rows == 8 * A.ck_lane && A.vec16 && A.ck_words <= A.W) {
            A.ck = const_cast<uint32_t *>(A.sig);
            A.ck_stride = A.W;
        } else {
            pack = true;
        }
    }
    uint32_t *ck = A.ck == A.sig ? nullptr : A.ck;
    int cur = 0;
    if (N <= kSmallObjs) {
        blsh_time_start(ctx, s);
        band_small_kernel<<<(unsigned)A.bands, 32 * kSmallWarps, 0, s>>>(A, key_bits, keys[0], vals[0], ck, pack);
        BLSH_LAUNCHED(ctx, "band_small_kernel");
    } else {
        // signature words a tile needs, and the rows that fit 40 KB
        int words = A.kind == BLSH_COSINE ? (A.rows * A.bands + 31) / 32 : A.rows * A.bands;
        int objs = 256;
        while (objs > 8 && objs * (words | 1) * 4 > 40 * 1024) objs >>= 1;
        if (objs * (words | 1) * 4 > 40 * 1024) words = 0;   // more than 1,280 words a row
        const size_t smem = words ? (size_t)objs * (words | 1) * 4 : 0;
        const long long tiles = (N + objs - 1) / objs, most = (long long)ctx->sm_count * 32;
        blsh_time_start(ctx, s);
        band_keys32_kernel<<<(unsigned)(tiles < most ? tiles : most), 256, smem, s>>>(A, keys[0], ck, words, objs, pack);
        BLSH_LAUNCHED(ctx, "band_keys_kernel");
        uint32_t *hist = keys[0] + n;
        const blsh_radix::Shape S = blsh_radix::shape(N, A.bands);
        // 27 bits of Jaccard keys: three digits of nine bits, not four of eight
        const int rc = (key_bits + 8) / 9 < (key_bits + 7) / 8
                           ? blsh_radix::sort_segments<uint32_t, 9>(ctx, keys, vals, S, key_bits, 0, true, hist,
                                                                    (uint32_t *)(ws + L.partial),
                                                                    (uint32_t *)(ws + L.grand), s, &cur)
                           : blsh_radix::sort_segments<uint32_t, 8>(ctx, keys, vals, S, key_bits, 0, true, hist,
                                                                    (uint32_t *)(ws + L.partial),
                                                                    (uint32_t *)(ws + L.grand), s, &cur);
        if (rc) return rc;
        if (A.exact_classes) {
            const unsigned grid = (unsigned)((n + 255) / 256 < 65535ll * 16 ? (n + 255) / 256 : 65535ll * 16);
            blsh_time_start(ctx, s);
            class_id_kernel<<<grid, 256, 0, s>>>(A, ck, keys[cur], vals[cur], n);
            BLSH_LAUNCHED(ctx, "class_id_kernel");
        }
    }
    const long long chunks = (n + 31) / 32;
    EmitState E;
    E.kept = (uint32_t *)(ws + L.counts);
    E.partners = keys[1] + n;
    E.chunk = (unsigned long long *)(ws + up256(L.counts + (size_t)n * 4));   // n / 4 bytes (into hist, unused here, for n < 71)
    E.rec_off = (unsigned long long *)(ws + L.rec_off);
    E.rec = (uint32_t *)(ws + L.rec);
    E.rec_cap = (workspace_bytes - L.rec) / 4;                // the keep record: the workspace past L.rec
    unsigned long long *work = &ctx->scratch->band_work[0];   // the passes' counters, the record's words, the tasks
    E.rec_next = work + 5;
    E.task_next = work + 6;
    E.tasks = (uint2 *)(ws + L.hist + 256);                   // (the chunk totals of a tiny n may reach into hist)
    E.task_cap = (L.partial - L.hist - 256) / sizeof(uint2);  // n / 32 of them
    // a chunk may be split: its partners end up to 31 positions past a whole
    // bucket of N, where the band begins on the chunk's last lane
    const bool long_walks = N + 30 > kSplit;
    E.next = work;
    int rc = emit_dispatch<kCount>(ctx, A, keys[cur], vals[cur], n, E, nullptr, 0, s);
    if (rc) return rc;
    if (long_walks) {
        E.next = work + 1;
        rc = emit_dispatch<kSegment>(ctx, A, keys[cur], vals[cur], n, E, nullptr, 0, s);
        if (rc) return rc;
    }
    rc = blsh_scan::run<unsigned long long>(ctx, E.chunk, E.chunk, chunks, (unsigned long long *)(ws + L.partial),
                                            (unsigned long long *)n_pairs, s);
    if (rc) return rc;
    const long long blocks = (n + 255) / 256, most = (long long)ctx->sm_count * 4;
    const unsigned grid = (unsigned)(blocks < most ? blocks : most);
    E.next = work + 2;
    blsh_time_start(ctx, s);
    emit_write_kernel<false><<<grid, 256, 0, s>>>(vals[cur], n, E, pairs, cap, (const long long *)n_pairs, ctx->scratch);
    BLSH_LAUNCHED(ctx, "emit_warp_kernel (write pass)");
    if (long_walks) {
        E.next = work + 3;
        blsh_time_start(ctx, s);
        emit_write_kernel<true><<<grid, 256, 0, s>>>(vals[cur], n, E, pairs, cap, (const long long *)n_pairs,
                                                     ctx->scratch);
        BLSH_LAUNCHED(ctx, "emit_warp_kernel (write pass, segments)");
    }
    E.next = work + 4;
    return emit_dispatch<kRetest>(ctx, A, keys[cur], vals[cur], n, E, pairs, cap, s);
}

// 64-bit keys with the band on top, sorted as a whole; emit_kernel.
int unstaged_candidates(blsh_ctx *ctx, const BandArgs &A, const Layout &L, char *ws, uint32_t *pairs, int64_t cap,
                        int64_t *n_pairs, cudaStream_t s) {
    const long long n = A.N * A.bands;
    unsigned long long *keys[2] = {(unsigned long long *)(ws + L.keys0), (unsigned long long *)(ws + L.keys1)};
    uint32_t *vals[2] = {(uint32_t *)(ws + L.vals0), (uint32_t *)(ws + L.vals1)};
    unsigned long long *counts = (unsigned long long *)(ws + L.counts);
    if (A.kind == BLSH_COSINE)   // pad lanes past the last band stay zero
        BLSH_CUDA(ctx, cudaMemsetAsync(A.ck, 0, (size_t)A.N * A.ck_words * 4, s));
    const unsigned grid = (unsigned)((n + 255) / 256 < 65535ll * 16 ? (n + 255) / 256 : 65535ll * 16);
    blsh_time_start(ctx, s);
    band_keys_kernel<<<grid, 256, 0, s>>>(A, keys[0], vals[0]);
    BLSH_LAUNCHED(ctx, "band_keys_kernel");
    const int key_bits = A.kind == BLSH_COSINE ? A.band_bits + A.rows : 64;
    int cur = 0;
    const int rc = blsh_radix::sort(ctx, keys, vals, n, key_bits, (uint32_t *)(ws + L.hist), (uint32_t *)(ws + L.partial),
                                    (uint32_t *)(ws + L.grand), s, &cur);
    if (rc) return rc;
    blsh_time_start(ctx, s);
    emit_kernel<false><<<grid, 256, 0, s>>>(A, keys[cur], vals[cur], n, counts, pairs, cap);
    BLSH_LAUNCHED(ctx, "emit_kernel (count pass)");
    const int rs = blsh_scan::run<unsigned long long>(ctx, counts, counts, n, (unsigned long long *)(ws + L.partial),
                                                      (unsigned long long *)n_pairs, s);
    if (rs) return rs;
    blsh_time_start(ctx, s);
    emit_kernel<true><<<grid, 256, 0, s>>>(A, keys[cur], vals[cur], n, counts, pairs, cap);
    BLSH_LAUNCHED(ctx, "emit_kernel (write pass)");
    blsh_time_start(ctx, s);
    check_cap_kernel<<<1, 1, 0, s>>>((const long long *)n_pairs, cap, ctx->scratch);
    BLSH_LAUNCHED(ctx, "check_cap_kernel");
    return BLSH_OK;
}

}  // namespace

extern "C" int blsh_lsh_candidates_workspace(int64_t N, int32_t kind, int32_t rows, int32_t bands, size_t *bytes) {
    if (!bytes || N < 0 || bands <= 0 || rows <= 0) return BLSH_EINVAL;
    if (kind != BLSH_JACCARD && kind != BLSH_COSINE) return BLSH_EINVAL;
    *bytes = layout(N, kind, rows, bands).total;
    return BLSH_OK;
}

extern "C" int blsh_lsh_candidates(blsh_ctx *ctx, const uint32_t *sig, int64_t N, int32_t sig_words, int32_t kind,
                                   int32_t rows, int32_t bands, uint32_t *pairs, int64_t cap, int64_t *n_pairs,
                                   void *workspace, size_t workspace_bytes, void *stream) {
    if (!ctx) return BLSH_EINVAL;
    if (!sig || !n_pairs || (cap > 0 && !pairs)) return blsh_fail(ctx, BLSH_EINVAL, "sig and n_pairs are required");
    if (kind != BLSH_JACCARD && kind != BLSH_COSINE) return blsh_fail(ctx, BLSH_EINVAL, "bad kind");
    if (N < 0 || N > (1ll << 32) || rows <= 0 || bands <= 0 || cap < 0)
        return blsh_fail(ctx, BLSH_EINVAL, "bad N, rows, bands or cap");
    if (kind == BLSH_COSINE && (rows > 32 || (long long)rows * bands > 32ll * sig_words))
        return blsh_fail(ctx, BLSH_EINVAL, "cosine bands need rows <= 32 and rows*bands <= 32*sig_words bits");
    if (kind == BLSH_JACCARD && (long long)rows * bands > sig_words)
        return blsh_fail(ctx, BLSH_EINVAL, "rows*bands exceeds the signature length");
    const int band_bits = band_bits_for(bands);
    if (kind == BLSH_COSINE && band_bits + rows > 64) return blsh_fail(ctx, BLSH_EINVAL, "too many bands");
    if ((long long)N * bands >= (1ll << 32)) return blsh_fail(ctx, BLSH_EINVAL, "N * bands must be < 2^32");
    if (!blsh_aligned(n_pairs, 8) || !blsh_aligned(workspace, 256) || !blsh_aligned(pairs, 8))
        return blsh_fail(ctx, BLSH_EINVAL, "misaligned pointer");
    const Layout L = layout(N, kind, rows, bands);
    if (!workspace || workspace_bytes < L.rec)
        return blsh_fail(ctx, BLSH_ETRUNC, "workspace needs %zu bytes", L.rec);
    blsh_device_guard g(ctx->device);
    cudaStream_t s = blsh_stream(stream);
    const long long n = N * bands;
    if (n == 0 || N < 2) {
        BLSH_CUDA(ctx, cudaMemsetAsync(n_pairs, 0, sizeof(int64_t), s));
        return BLSH_OK;
    }
    char *ws = (char *)workspace;
    BandArgs A;
    A.sig = sig;
    A.N = N;
    A.W = sig_words;
    A.kind = kind;
    A.rows = rows;
    A.bands = bands;
    A.band_bits = band_bits;
    A.key_shift = 64 - band_bits;
    A.exact_classes = kind == BLSH_JACCARD && jac_row_words(bands) <= kStageWords;
    A.bk = kind == BLSH_JACCARD && !A.exact_classes ? (unsigned long long *)(ws + L.bk) : nullptr;
    A.ck = kind == BLSH_COSINE || A.exact_classes ? (uint32_t *)(ws + L.ck) : nullptr;
    A.ck_lane = A.exact_classes ? 4 : cos_lane_bytes(rows);
    A.vec16 = blsh_aligned(sig, 16) && sig_words % 4 == 0;
    A.ck_words = A.exact_classes ? jac_row_words(bands) : cos_row_words(rows, bands);
    A.ck_stride = A.ck_words;
    const bool staged = (kind == BLSH_COSINE || A.exact_classes) && A.ck_words <= kStageWords;
    BLSH_CUDA(ctx, cudaMemsetAsync(&ctx->scratch->band_work[0], 0, sizeof(ctx->scratch->band_work), s));
    return staged ? staged_candidates(ctx, A, L, ws, workspace_bytes, pairs, cap, n_pairs, s)
                  : unstaged_candidates(ctx, A, L, ws, pairs, cap, n_pairs, s);
}
