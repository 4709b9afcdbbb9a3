// lite.cu -- Algorithm 2 (BayesLSH-Lite).
//
// Pass 1 is the verification kernel of verify.cu in its Lite form: the
// pruning loop over at most h hashes, no concentration test; an unpruned
// pair is marked as a survivor in its status byte.  Pass 2 (this file) gives
// every survivor its exact similarity: the survivors are collected into a
// queue (one atomic per 4 or 16 tiles of 512 statuses) and warps take batches
// of up to 32 from a counter, so the many survivors of one bucket of
// near-duplicates spread over the GPU; a warp intersects a batch's sorted
// index lists together, the elements of the shorter rows dealt over its lanes
// and searched in the longer ones in shared memory (lite_flat), or a few
// survivors one by one (lite_few).  Survivors beyond the queue's capacity are
// found by a scan of the statuses in tiles handed out by a counter.
//
//   Jaccard: s = |A n B| / |A u B|, one FP64 division.
//   Cosine:  s = D / sqrt(Nx * Ny) with D = sum over common indices of
//            rn(x_i * y_i * 2^60), Nx = sum rn(x_i^2 * 2^60), Ny likewise,
//            each term the exact product of two floats rounded to an
//            integer (formed with integer arithmetic) and added in int64, so
//            the sums do not depend on the order the lanes add them in.
// A pair is kept iff s > t.
#include <type_traits>

#include "verify.cuh"

namespace {

constexpr unsigned kFull = 0xffffffffu;

struct LiteArgs {
    const uint2 *pairs;
    long long P;
    const long long *P_dev;
    const int64_t *indptr;
    const uint32_t *indices;
    const float *values;
    double t;
    uint8_t *status;
    double *sim;
    blsh_dev_scratch *scratch;
    int vec;                  // status is 16-byte aligned
    long long N;
    const long long *norm2;   // cosine: each row's sum of fixed_term(v, v), or NULL (formed per pair)
};

constexpr int kLiteGrab = 16;   // tiles of 512 statuses per grab (this pass sees only survivors the queue missed)

// rn(u v 2^60) for two floats, by integer arithmetic: u = mu 2^eu and
// v = mv 2^ev with 24-bit integer mantissas, so u v 2^60 = mu mv 2^(eu+ev+60)
// and the 48-bit product is shifted with round-half-to-even (symmetric, as
// the FP64 conversion rounds).  The same value as the FP64 expression
// rn((double)u * (double)v * 2^60) (the product of two floats is exact in
// FP64).  Products of |u v| >= 2^2 (outside rows of squared norm below 4)
// are shifted up as far as they fit and otherwise saturate to the int64
// limit of their sign, as that conversion does; non-finite inputs saturate
// by sign.  All integer arithmetic: the FP64 pipe is narrow on this part,
// and a branch to FP64 code here was executed (predicated) for every term.
__device__ __forceinline__ long long fixed_term(float u, float v) {
    const uint32_t bu = __float_as_uint(u), bv = __float_as_uint(v);
    int eu = (int)((bu >> 23) & 0xffu), ev = (int)((bv >> 23) & 0xffu);
    uint32_t mu = bu & 0x7fffffu, mv = bv & 0x7fffffu;
    if (eu) mu |= 0x800000u; else eu = 1;   // subnormals: exponent 1 - 150
    if (ev) mv |= 0x800000u; else ev = 1;
    const unsigned long long prod = (unsigned long long)mu * mv;   // < 2^48
    const int sh = eu + ev - 300 + 60;                               // u v 2^60 = prod 2^sh
    unsigned long long r;
    if (sh >= 0) {
        if (sh > 15 && (sh >= 63 || (prod >> (63 - sh)) != 0))   // at least 2^63 in magnitude
            return ((bu ^ bv) >> 31) ? (long long)0x8000000000000000ull : 0x7fffffffffffffffll;
        r = prod << sh;
    } else if (-sh > 48) {
        r = 0;                                                       // below half of 2^0
    } else {
        const int k = -sh;
        const unsigned long long q = prod >> k, rem = prod & ((1ull << k) - 1ull), half = 1ull << (k - 1);
        r = q + ((rem > half || (rem == half && (q & 1ull))) ? 1ull : 0ull);
    }
    return ((bu ^ bv) >> 31) ? -(long long)r : (long long)r;
}

// fixed_term(v, v) with one rounded shift where v lies in the range of a unit
// vector's entries: the product, moved up 15 bits, is shifted down by 1 to 63.
__device__ __forceinline__ long long fixed_square(float v) {
    const uint32_t b = __float_as_uint(v) & 0x7fffffffu;
    uint32_t e = b >> 23, m = b & 0x7fffffu;
    if (e) m |= 0x800000u; else e = 1;
    const int down = 15 - (2 * (int)e - 240);
    if (down < 1 || down > 63) return fixed_term(v, v);
    const unsigned long long t = ((unsigned long long)m * m) << 15;
    return (long long)((t + ((1ull << (down - 1)) - 1ull) + ((t >> down) & 1ull)) >> down);   // half to even
}

__device__ __forceinline__ long long warp_sum(long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// First position in L[0..n) holding a value >= v (L in global or shared
// memory).
__device__ __forceinline__ long long lower_bound(const uint32_t *L, long long n, uint32_t v) {
    long long lo = 0, hi = n;
    while (lo < hi) {
        const long long mid = (lo + hi) >> 1;
        if (L[mid] < v) lo = mid + 1; else hi = mid;
    }
    return lo;
}

constexpr int kLiteStage = 512;   // half the elements a warp stages in shared memory

// The sums of one survivor's exact similarity (the whole warp): rows
// x = [ax, ax+na) and y = [ay, ay+nb) of the CSR; D_out = the intersection
// size (sets) or D (cosine), and for cosine without have_norms the two
// squared norms.  The shorter row's elements are spread over the lanes and each
// is looked up in the longer row by binary search: with the longer row held
// one element per lane (at most 32 elements: the search steps are shuffles),
// staged in the warp's shared memory, a tile at a time.  (Searching rows of
// more than 512 elements in global memory, two lookups in flight, took 62 us
// for 3,600 survivors whose longest rows have some 900 elements; 42 now.)
// KEEP: x's elements are looked up in y, whichever is shorter.
template <bool COSINE, bool KEEP = false>
__device__ __forceinline__ void lite_exact_one(const LiteArgs &A, long long ax, long long na, long long ay,
                                               long long nb, bool have_norms, uint32_t *w_idx,
                                               long long &D_out, long long &Nx_out, long long &Ny_out) {
    const int lane = threadIdx.x & 31;
    // the shorter row S, the longer row L (the sums below do not depend on
    // which row is which)
    long long s0 = ax, ns = na, l0 = ay, nl = nb;
    if (!KEEP && nb < na) { s0 = ay; ns = nb; l0 = ax; nl = na; }
    long long inter = 0, D = 0, Ns = 0, Nl = 0;
    if (!KEEP && nl <= 32) {
        // lane e holds element e of both rows
        uint32_t si = 0, li = 0;
        float sv = 0.0f, lv = 0.0f;
        if (lane < ns) {
            si = __ldg(A.indices + s0 + lane);
            if (COSINE) sv = __ldg(A.values + s0 + lane);
        }
        if (lane < nl) {
            li = __ldg(A.indices + l0 + lane);
            if (COSINE) lv = __ldg(A.values + l0 + lane);
        }
        // first position p of L with L[p] >= si: at most 32 candidates, so six
        // halvings of [lo, hi) settle every lane
        int lo = 0, hi = (int)nl;
#pragma unroll
        for (int it = 0; it < 6; ++it) {
            const int mid = (lo + hi) >> 1;
            const uint32_t v = __shfl_sync(kFull, li, mid & 31);
            if (lo < hi) {
                if (v < si) lo = mid + 1;
                else hi = mid;
            }
        }
        const uint32_t at = __shfl_sync(kFull, li, lo & 31);
        const bool hit = lane < ns && lo < nl && at == si;
        if (!COSINE) {
            inter = __popc(__ballot_sync(kFull, hit));
        } else {
            const float atv = __shfl_sync(kFull, lv, lo & 31);
            D = hit ? fixed_term(sv, atv) : 0;
            if (!have_norms) {
                Ns = lane < ns ? fixed_term(sv, sv) : 0;
                Nl = lane < nl ? fixed_term(lv, lv) : 0;
            }
        }
    } else {
        // the longer row's indices through the warp's stage, kTile at a time;
        // the shorter row's elements up to the tile's last are looked up in it
        // four per lane (their loads, searches and values overlap: a warp that
        // forms one survivor has nothing else to wait behind)
        constexpr int kTile = 2 * kLiteStage;
        long long sp = 0;                                  // the shorter row's elements done
        if (KEEP && COSINE && !have_norms && nl == 0)      // no tile to look them up in
            for (long long i = lane; i < ns; i += 32) {
                const float v = __ldg(A.values + s0 + i);
                Ns += fixed_term(v, v);
            }
        for (long long tb = 0; tb < nl && (sp < ns || (COSINE && !have_norms)); tb += kTile) {
            const int tn = (int)(nl - tb < kTile ? nl - tb : kTile);
            __syncwarp();                                  // the previous tile is done with the stage
#pragma unroll 4
            for (int i = lane; i < tn; i += 32) w_idx[i] = __ldg(A.indices + l0 + tb + i);
            if (COSINE && !have_norms)
#pragma unroll 4
                for (int i = lane; i < tn; i += 32) {
                    const float v = __ldg(A.values + l0 + tb + i);
                    Nl += fixed_term(v, v);
                }
            __syncwarp();
            const uint32_t last = w_idx[tn - 1];
            const bool final_tile = tb + tn >= nl;
            // U elements a lane against a tile of fewer than 2 TOP
            auto round = [&](auto width, auto top) {
                constexpr int U = decltype(width)::value, TOP = decltype(top)::value;
                uint32_t v[U];
                bool in[U];
                int pos[U];
                unsigned taken = 0;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const long long i = sp + 32 * u + lane;
                    v[u] = i < ns ? __ldg(A.indices + s0 + i) : 0u;
                    in[u] = i < ns && (final_tile || v[u] <= last);
                    pos[u] = 0;
                }
#pragma unroll
                for (int u = 0; u < U; ++u) taken += __popc(__ballot_sync(kFull, in[u]));
                for (int step = TOP; step > 0; step >>= 1)
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (pos[u] + step <= tn && w_idx[pos[u] + step - 1] < v[u]) pos[u] += step;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const bool hit = in[u] && pos[u] < tn && w_idx[pos[u]] == v[u];
                    if (!COSINE) {
                        inter += hit;
                    } else {
                        const long long i = s0 + sp + 32 * u + lane;
                        const float sv = in[u] && (hit || !have_norms) ? __ldg(A.values + i) : 0.0f;
                        if (hit) D += fixed_term(sv, __ldg(A.values + l0 + tb + pos[u]));
                        if (!have_norms && in[u]) Ns += fixed_term(sv, sv);
                    }
                }
                sp += taken;
                return taken == 32 * U && sp < ns;         // the rest lies past this tile, or none is left
            };
            if (!KEEP && tn < 128 && ns - sp <= 64) {
                if (sp < ns) round(std::integral_constant<int, 2>{}, std::integral_constant<int, 64>{});
            } else {
                for (bool more = sp < ns; more;)
                    more = round(std::integral_constant<int, 4>{}, std::integral_constant<int, kTile / 2>{});
            }
        }
    }
    // the warp's sums (the same in every lane): the intersection size, or D
    // and the two squared norms (which row is which does not matter: the
    // similarity uses their product)
    if (!COSINE) {
        D_out = KEEP || nl > 32 ? warp_sum(inter) : inter;
    } else {
        D_out = warp_sum(D);
        if (!have_norms) {
            Nx_out = warp_sum(Ns);
            Ny_out = warp_sum(Nl);
        }
    }
}

// The sums of up to 32 / W survivors at once, each in its own W-lane
// segment of the warp (W = 8 or 16), for survivors whose two rows have at
// most W elements each: the register path of lite_exact_one with the
// shuffles, the search and the sums kept inside the segment.  sel holds the
// lanes whose survivors are to be formed; lane i's survivor rows are
// [ax, ex) and [ay, ey) in lane i.  Segment k takes the k-th survivor left
// in sel; each survivor's lane receives its sums.
template <bool COSINE, int W>
__device__ __forceinline__ void lite_segments(const LiteArgs &A, unsigned sel, long long ax, long long ex,
                                              long long ay, long long ey, bool have_norms, long long &myD,
                                              long long &myNx, long long &myNy) {
    constexpr int S = 32 / W;
    const int lane = threadIdx.x & 31;
    const int e = lane & (W - 1), seg = lane / W;
    const unsigned lt = (1u << lane) - 1u;
    while (sel) {
        // the first S survivors left: segment seg takes the seg-th of them
        unsigned taken = sel, rest = sel;
#pragma unroll
        for (int k = 0; k < S; ++k) rest &= rest - 1;
        taken &= ~rest;
        unsigned m = taken;
        for (int k = 0; k < seg && m; ++k) m &= m - 1;
        const int pick = m ? __ffs(m) - 1 : -1;
        const int src = pick < 0 ? 0 : pick;
        const long long a0 = __shfl_sync(kFull, ax, src), a1 = __shfl_sync(kFull, ex, src);
        const long long b0 = __shfl_sync(kFull, ay, src), b1 = __shfl_sync(kFull, ey, src);
        long long s0 = a0, ns = a1 - a0, l0 = b0, nl = b1 - b0;
        if (nl < ns) { s0 = b0; ns = b1 - b0; l0 = a0; nl = a1 - a0; }
        if (pick < 0) ns = nl = 0;
        uint32_t si = 0, li = 0;
        float sv = 0.0f, lv = 0.0f;
        if (e < ns) {
            si = __ldg(A.indices + s0 + e);
            if (COSINE) sv = __ldg(A.values + s0 + e);
        }
        if (e < nl) {
            li = __ldg(A.indices + l0 + e);
            if (COSINE) lv = __ldg(A.values + l0 + e);
        }
        // first position p of L with L[p] >= si, among 0..nl (nl <= W)
        int lo = 0, hi = (int)nl;
#pragma unroll
        for (int it = 0; (1 << it) <= W; ++it) {
            const int mid = (lo + hi) >> 1;
            const uint32_t v = __shfl_sync(kFull, li, mid & (W - 1), W);
            if (lo < hi) {
                if (v < si) lo = mid + 1;
                else hi = mid;
            }
        }
        const uint32_t at = __shfl_sync(kFull, li, lo & (W - 1), W);
        const bool hit = e < ns && lo < nl && at == si;
        long long D = 0, Ns = 0, Nl = 0;
        if (!COSINE) {
            const unsigned segmask = (W == 32 ? kFull : ((1u << W) - 1u)) << (seg * W);
            D = __popc(__ballot_sync(kFull, hit) & segmask);
        } else {
            const float atv = __shfl_sync(kFull, lv, lo & (W - 1), W);
            D = hit ? fixed_term(sv, atv) : 0;
            if (!have_norms) {
                Ns = e < ns ? fixed_term(sv, sv) : 0;
                Nl = e < nl ? fixed_term(lv, lv) : 0;
            }
#pragma unroll
            for (int o = W / 2; o > 0; o >>= 1) {
                D += __shfl_xor_sync(kFull, D, o);
                if (!have_norms) {
                    Ns += __shfl_xor_sync(kFull, Ns, o);
                    Nl += __shfl_xor_sync(kFull, Nl, o);
                }
            }
        }
        // survivor i's sums from the first lane of its segment
        const int from = W * __popc(taken & lt);
        const long long gD = __shfl_sync(kFull, D, from & 31);
        const long long gNs = __shfl_sync(kFull, Ns, from & 31), gNl = __shfl_sync(kFull, Nl, from & 31);
        if ((taken >> lane) & 1u) {
            myD = gD;
            if (COSINE && !have_norms) {
                myNx = gNs;
                myNy = gNl;
            }
        }
        sel = rest;
    }
}

// The similarity from the sums (one lane per survivor: FP64 is a narrow
// pipe on this part, so the division and square root run once per survivor
// rather than once per lane of a warp-wide computation).
template <bool COSINE>
__device__ __forceinline__ double lite_similarity(long long D, long long Nx, long long Ny, long long na,
                                                  long long nb) {
    if (!COSINE) {
        const long long uni = na + nb - D;
        return uni == 0 ? 0.0 : __ddiv_rn((double)D, (double)uni);
    }
    if (Nx == 0 || Ny == 0) return 0.0;
    return __ddiv_rn(__ll2double_rn(D), __dsqrt_rn(__dmul_rn(__ll2double_rn(Nx), __ll2double_rn(Ny))));
}

// The sums of a batch of survivors (this lane's, if `mine`: rows [ax, ex) and
// [ay, ey), each below 2^26 elements), the elements of their shorter rows dealt over the
// lanes: element t of the batch goes to lane t mod 32, whatever survivor it
// belongs to, and is looked up in that survivor's longer row by binary search
// -- in shared memory where that row has at most kFlatStage elements and the
// batch's rows fit the stage (copied asynchronously, all at once), in global
// memory otherwise.  Hits are listed, and 32 at a time read their values and
// add their terms to the survivors' sums in shared memory, in three limbs of
// 24, 24 and 16 bits (32-bit adds are native there), carried into a 64-bit sum
// before they can overflow.
// A warp per survivor spent 430 issue slots on each (broadcasts of the bounds,
// a search of six shuffle rounds and a 64-bit reduction over 32 lanes, for 8.9
// elements on average).  4.6e7 survivors of 5e6 documents: 16.7 ms, 10.0
// here.
constexpr int kFlatStage = 127;    // (seven halvings)
constexpr int kFlatMin = 8;        // survivors in a batch from which it is formed this way
constexpr int kFlatCarry = 8;      // hit rounds (of 32) between carries: 256 times 2^24 - 1 fits a limb
// a warp's limbs [3][32], rows [32] uint4, lengths [32] uint2, hits [64] uint2, in words
constexpr int kFlatWords = 96 + 128 + 64 + 128;

__device__ __forceinline__ void copy16_async(uint32_t *dst, const uint32_t *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

template <bool COSINE>
__device__ __forceinline__ long long lite_flat(const LiteArgs &A, bool mine, long long ax, long long ex, long long ay,
                                               long long ey, long long nnz, uint32_t *stage, uint32_t *flat) {
    const int lane = threadIdx.x & 31;
    uint32_t *limbs = flat;
    uint4 *rows = reinterpret_cast<uint4 *>(flat + 96);            // [32]: first elements of S and L
    uint2 *lens = reinterpret_cast<uint2 *>(flat + 96 + 128);      // [32]: |L|, its place in the stage (~0: none)
    uint2 *hits = lens + 32;                                       // [64]: owner | element of S << 5, element of L
    long long s0 = ax, l0 = ay;
    unsigned ns = mine ? (unsigned)(ex - ax) : 0u, nl = mine ? (unsigned)(ey - ay) : 0u;
    if (nl < ns) {
        s0 = ay;
        l0 = ax;
        const unsigned t = ns;
        ns = nl;
        nl = t;
    }
    // staged rows: those of up to kFlatStage elements, while they fit (copied
    // in whole 16-byte blocks, which must lie inside the index array); their
    // survivors come first, so that few rounds mix the two kinds of lookup
    const unsigned phase = ((unsigned)((uintptr_t)(A.indices + l0) >> 2)) & 3u;   // words into its block
    const unsigned blocks = (phase + nl + 3) >> 2;
    const bool fits = nl != 0 && nl <= kFlatStage && l0 - phase >= 0 && l0 - phase + 4ll * blocks <= nnz;
    const unsigned want = fits ? 4 * blocks : 0u;
    const unsigned lt = (1u << lane) - 1u;
    unsigned at = want;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned v = __shfl_up_sync(kFull, at, o);
        if (lane >= o) at += v;
    }
    const bool staged = want != 0 && at <= 2 * kLiteStage;
    const unsigned sm = __ballot_sync(kFull, staged);
    const int slot = staged ? __popc(sm & lt) : __popc(sm) + __popc(~sm & lt);
    __syncwarp();                                  // the previous batch is done with the stage and the limbs
    limbs[slot] = ns;
    rows[slot] = make_uint4((unsigned)s0, (unsigned)(s0 >> 32), (unsigned)l0, (unsigned)(l0 >> 32));
    lens[slot] = make_uint2(nl, staged ? at - want + phase : ~0u);
    __syncwarp();
    const unsigned slot_ns = limbs[lane];
    unsigned off = slot_ns;                        // the slot's first element in the batch
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned v = __shfl_up_sync(kFull, off, o);
        if (lane >= o) off += v;
    }
    const unsigned total = __shfl_sync(kFull, off, 31);
    off -= slot_ns;
    limbs[lane] = limbs[32 + lane] = limbs[64 + lane] = 0;
    __syncwarp();
    // four rows at a time, eight lanes and 128 bytes each
    const int n_staged = __popc(sm);
#pragma unroll 1
    for (int r = lane >> 3; r < n_staged; r += 4) {
        const uint2 ln = lens[r];
        const uint4 rw = rows[r];
        const unsigned ph = ln.y & 3u, nb = (ph + ln.x + 3) >> 2;   // stage places start on 16 bytes, plus phase
        const uint32_t *src = A.indices + (((long long)rw.w << 32 | rw.z) - ph);
        uint32_t *dst = stage + (ln.y - ph);
#pragma unroll 1
        for (unsigned e = lane & 7; e < nb; e += 8) copy16_async(dst + 4 * e, src + 4 * e);
    }
    long long D = 0;
    auto carry = [&]() {                           // the limbs into the slot's sum (lane = slot)
        __syncwarp();
        D += (long long)limbs[lane];
        if (COSINE)
            D += (long long)(((unsigned long long)limbs[32 + lane] << 24) +
                             ((unsigned long long)(long long)(int)limbs[64 + lane] << 48));
        limbs[lane] = limbs[32 + lane] = limbs[64 + lane] = 0;
        __syncwarp();
    };
    // the terms of hits [h0, h0 + m), a lane each
    unsigned rounds = 0;
    auto add_hits = [&](int h0, int m) {
        __syncwarp();
        if (lane < m) {
            const uint2 h = hits[h0 + lane];
            const int o = (int)(h.x & 31u);
            if (COSINE) {
                const uint4 rw = rows[o];
                const long long term = fixed_term(__ldg(A.values + ((long long)rw.y << 32 | rw.x) + (h.x >> 5)),
                                                  __ldg(A.values + ((long long)rw.w << 32 | rw.z) + h.y));
                atomicAdd(limbs + o, (uint32_t)term & 0xffffffu);
                atomicAdd(limbs + 32 + o, (uint32_t)((unsigned long long)term >> 24) & 0xffffffu);
                atomicAdd(limbs + 64 + o, (uint32_t)(int)(term >> 48));
            } else {
                atomicAdd(limbs + o, 1u);
            }
        }
        if (++rounds % kFlatCarry == 0) carry();
    };
    // element t of the batch: its survivor, its place there and its value (the
    // next round's are loaded before this round's are looked up)
    auto element = [&](unsigned t, int &o, unsigned &e, uint32_t &v) {
        o = 0;                                     // the last lane whose offset is <= t
#pragma unroll
        for (int step = 16; step > 0; step >>= 1) {
            const unsigned oc = __shfl_sync(kFull, off, o + step);
            if (oc <= t) o += step;
        }
        e = t - __shfl_sync(kFull, off, o);
        v = 0;
        if (t < total) {
            const uint4 rw = rows[o];
            v = __ldg(A.indices + ((long long)rw.y << 32 | rw.x) + e);
        }
    };
    int o;
    unsigned e;
    uint32_t v;
    element(lane, o, e, v);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    int n_hits = 0;
    for (unsigned t0 = 0; t0 < total; t0 += 32) {
        int o2 = 0;
        unsigned e2 = 0;
        uint32_t v2 = 0;
        if (t0 + 32 < total) element(t0 + 32 + lane, o2, e2, v2);
        bool hit = false;
        unsigned lo = 0;
        if (t0 + lane < total) {
            const uint2 ln = lens[o];
            // lo = the elements of L below v, by halving steps without branches
            if (ln.y != ~0u) {
                const uint32_t *L = stage + ln.y;
#pragma unroll
                for (unsigned step = (kFlatStage + 1) / 2; step > 0; step >>= 1)
                    if (lo + step <= ln.x && L[lo + step - 1] < v) lo += step;
                hit = lo < ln.x && L[lo] == v;
            } else {
                const uint4 rw = rows[o];
                const uint32_t *L = A.indices + ((long long)rw.w << 32 | rw.z);
                for (unsigned step = ln.x ? 1u << (31 - __clz(ln.x)) : 0u; step > 0; step >>= 1)
                    if (lo + step <= ln.x && __ldg(L + lo + step - 1) < v) lo += step;
                hit = lo < ln.x && __ldg(L + lo) == v;
            }
        }
        const unsigned hm = __ballot_sync(kFull, hit);
        if (COSINE && hit) {                       // the values it will read, on their way meanwhile
            const uint4 rw = rows[o];
            asm volatile("prefetch.global.L2 [%0];" ::"l"(A.values + ((long long)rw.y << 32 | rw.x) + e));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(A.values + ((long long)rw.w << 32 | rw.z) + lo));
        }
        if (hit) hits[n_hits + __popc(hm & ((1u << lane) - 1u))] = make_uint2((unsigned)o | e << 5, lo);
        n_hits += __popc(hm);
        if (n_hits >= 32) {
            n_hits -= 32;
            add_hits(n_hits, 32);
        }
        o = o2;
        e = e2;
        v = v2;
    }
    if (n_hits) add_hits(0, n_hits);
    carry();
    return __shfl_sync(kFull, D, slot);
}

struct LiteSums {
    long long D, Nx, Ny;
};

// The sums of the survivors of the lanes in `todo`, segments of the warp or the
// whole warp on each; Nx and Ny as they come in when the norms are formed.
template <bool COSINE>
__device__ __forceinline__ LiteSums lite_few(const LiteArgs &A, unsigned todo, long long ax, long long ex, long long ay,
                                          long long ey, bool have_norms, LiteSums in, uint32_t *w_idx) {
    const int lane = threadIdx.x & 31;
    LiteSums my = in;
    // survivors whose rows are short share the warp: four at a time when
    // both rows have at most 8 elements, two when at most 16 (a group too
    // small to fill the segments joins the next wider one)
    const long long longest = ex - ax > ey - ay ? ex - ax : ey - ay;
    unsigned s8 = __ballot_sync(kFull, longest <= 8) & todo;
    unsigned s16 = __ballot_sync(kFull, longest <= 16) & ~s8 & todo;
    if (__popc(s8) < 3) {
        s16 |= s8;
        s8 = 0u;
    }
    if (__popc(s16) < 2) s16 = 0u;
    if (s8) lite_segments<COSINE, 8>(A, s8, ax, ex, ay, ey, have_norms, my.D, my.Nx, my.Ny);
    if (s16) lite_segments<COSINE, 16>(A, s16, ax, ex, ay, ey, have_norms, my.D, my.Nx, my.Ny);
    for (todo &= ~(s8 | s16); todo; todo &= todo - 1) {
        const int i = __ffs(todo) - 1;
        const long long a0 = __shfl_sync(kFull, ax, i), a1 = __shfl_sync(kFull, ex, i);
        const long long b0 = __shfl_sync(kFull, ay, i), b1 = __shfl_sync(kFull, ey, i);
        long long D = 0, Nx = 0, Ny = 0;
        lite_exact_one<COSINE>(A, a0, a1 - a0, b0, b1 - b0, have_norms, w_idx, D, Nx, Ny);
        if (lane == i) {
            my.D = D;
            if (!have_norms) {
                my.Nx = Nx;
                my.Ny = Ny;
            }
        }
    }
    return my;
}

// Up to 32 survivors, survivor my_q of lane l (-1: none): their pairs, row
// bounds and (when formed) squared norms are loaded by all lanes at once, so
// those dependent loads overlap across the batch; then the warp forms their
// sums, and finally every lane turns its own survivor's sums into the
// similarity and writes it with the verdict.
//
// heavy (or NULL): survivors both of whose rows have more than kLiteHeavy
// elements are put there instead, while it has room, for lite_heavy: one of
// them takes a warp as long as dozens of batches, and a batch of 32 (a long row's
// survivors follow each other) held its warp 0.3 ms after all others had
// ended (a search over 6e5 vectors: queue 478 us, with the list 202 + 38; 256
// elements 184 + 39, 1,024 237 + 37).
// Their status is set apart from a survivor's until lite_heavy writes the
// verdict, so that the scan for survivors beyond the queue, which other CTAs
// run meanwhile, does not take them again.
constexpr int kLiteHeavy = 512;
constexpr uint8_t kHeavyStatus = 251;
static_assert(kHeavyStatus != BLSH_LITE_SURVIVOR && kHeavyStatus != BLSH_NEEDS_HASHES && kHeavyStatus != BLSH_BAD_PAIR,
              "the listed pairs' status must differ from every other status");
template <bool COSINE>
__device__ __forceinline__ void lite_batch(const LiteArgs &A, long long my_q, bool have_norms, uint32_t *w_idx,
                                           uint32_t *flat, unsigned long long *heavy = nullptr) {
    long long ax = 0, ex = 0, ay = 0, ey = 0;
    LiteSums my = {0, 0, 0};
    if (my_q >= 0) {
        const uint2 pr = __ldg(A.pairs + my_q);
        ax = __ldg(A.indptr + pr.x);
        ex = __ldg(A.indptr + pr.x + 1);
        ay = __ldg(A.indptr + pr.y);
        ey = __ldg(A.indptr + pr.y + 1);
        if (have_norms) {
            my.Nx = __ldg(A.norm2 + pr.x);
            my.Ny = __ldg(A.norm2 + pr.y);
        }
    }
    if (heavy && ex - ax > kLiteHeavy && ey - ay > kLiteHeavy) {
        const unsigned long long slot = atomicAdd(&A.scratch->recheck_count, 1ull);
        if (slot < BLSH_RECHECK_CAP) {
            heavy[slot] = (unsigned long long)my_q;
            A.status[my_q] = kHeavyStatus;
            my_q = -1;
        }
    }
    unsigned todo = __ballot_sync(kFull, my_q >= 0);
    if ((!COSINE || have_norms) && __popc(todo) >= kFlatMin) {
        // rows of 2^26 elements and more are left to lite_few
        const bool mine = my_q >= 0 && ((ex - ax) | (ey - ay)) < (1ll << 26);
        my.D = lite_flat<COSINE>(A, mine, ax, ex, ay, ey, __ldg(A.indptr + A.N), w_idx, flat);
        todo &= ~__ballot_sync(kFull, mine);
    }
    if (todo) my = lite_few<COSINE>(A, todo, ax, ex, ay, ey, have_norms, my, w_idx);
    if (my_q >= 0) {
        const double s = lite_similarity<COSINE>(my.D, my.Nx, my.Ny, ex - ax, ey - ay);
        A.sim[my_q] = s;
        A.status[my_q] = s > A.t ? BLSH_LITE_ACCEPT : BLSH_LITE_REJECT;
    }
}

// Each row's sum of fixed_term(v, v) (the squared norm of the exact cosine,
// an integer: independent of the order of the terms).  Eight lanes per row,
// four rows a warp; the lanes' sums meet in three shuffle steps.  (A warp over
// 128 consecutive elements with a search for every element's row and a
// segmented scan took 147 instructions per 32 elements: 1.27 ms for 1.4e8
// nonzeros; eight lanes for the longest rows too, 0.97; 0.56 here.)  Formed only when there are more survivors than
// half the rows (the collection pass has counted them); otherwise each
// survivor forms its two norms itself, which is less work.
constexpr int kNormLong = 256;   // (a row of 30,000 took eight lanes longer than all the others together)
__global__ void __launch_bounds__(256) row_norm2_kernel(const int64_t *__restrict__ indptr,
                                                        const float *__restrict__ values, long long N,
                                                        long long *__restrict__ norm2,
                                                        blsh_dev_scratch *scratch) {
    const bool form = scratch->work3 * 2ull > (unsigned long long)N;
    if (blockIdx.x == 0 && threadIdx.x == 0) scratch->norm2_valid = form ? 1u : 0u;
    if (!form) return;
    const int g = threadIdx.x & 7;
    const long long stride = (long long)gridDim.x * (blockDim.x >> 3);
    // (the trip count is the same for the whole warp)
    const long long first = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 3;
    for (long long w0 = first & ~3ll; w0 < N; w0 += stride) {
        const long long row = w0 + (first & 3);
        long long s = 0, e = 0;
        if (row < N) {
            s = __ldg(indptr + row);
            e = __ldg(indptr + row + 1);
        }
        long long sum = 0;
        // long rows: all of the warp's lanes, eight loads each
        const bool is_long = e - s > kNormLong;
        for (unsigned rows = __ballot_sync(kFull, is_long && g == 0); rows; rows &= rows - 1) {
            const int from = __ffs(rows) - 1;
            const long long ls = __shfl_sync(kFull, s, from), le = __shfl_sync(kFull, e, from);
            long long part = 0;
            for (long long i = ls + (threadIdx.x & 31); i < le; i += 256) {
                float v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = i + 32 * u < le ? __ldg(values + i + 32 * u) : 0.0f;
#pragma unroll
                for (int u = 0; u < 8; ++u) part += fixed_square(v[u]);   // (0 past the end)
            }
            part = warp_sum(part);
            if ((int)(threadIdx.x & 31) == from) sum = part;
        }
        if (is_long) s = e;
        for (long long i = s + g; i < e; i += 32) {
            float v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = i + 8 * u < e ? __ldg(values + i + 8 * u) : 0.0f;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (i + 8 * u < e) sum += fixed_square(v[u]);
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
        if (g == 0 && row < N) norm2[row] = sum;
    }
}

// per warp: the staging area (4 KB), lite_flat's area, a survivor list (a tile's 512 and up to 31 before them)
constexpr int kLiteWarpWords = 2 * kLiteStage + kFlatWords + 272;
static_assert(kLiteWarpWords % 4 == 0, "16-byte rows");

// The listed survivors of two long rows, a CTA each: warp w takes the w-th eighth
// of the shorter row and the part of the longer one that its elements can lie
// in (the parts cover it), and the warps' sums are added.
template <bool COSINE>
__device__ __forceinline__ void lite_heavy(const LiteArgs &A, const unsigned long long *heavy, bool have_norms,
                                           uint32_t *w_idx) {
    __shared__ long long s_sum[8][3];
    __shared__ unsigned long long s_item;
    const int warp = threadIdx.x >> 5;
    const unsigned long long listed = A.scratch->recheck_count;
    const unsigned long long n = listed < BLSH_RECHECK_CAP ? listed : BLSH_RECHECK_CAP;
    if (n == 0) return;
    for (;;) {
        __syncthreads();                                   // the previous survivor's sums have been read
        if (threadIdx.x == 0) s_item = atomicAdd(&A.scratch->hash_work, 1ull);
        __syncthreads();
        if (s_item >= n) break;
        const long long q = (long long)heavy[s_item];
        const uint2 pr = __ldg(A.pairs + q);
        const long long ax = __ldg(A.indptr + pr.x), na = __ldg(A.indptr + pr.x + 1) - ax;
        const long long ay = __ldg(A.indptr + pr.y), nb = __ldg(A.indptr + pr.y + 1) - ay;
        const bool swap = nb < na;
        const long long s0 = swap ? ay : ax, ns = swap ? nb : na, l0 = swap ? ax : ay, nl = swap ? na : nb;
        // where this warp's parts of the two rows begin, and the next one's (equal indices stay together)
        long long at[2], cut[2];
#pragma unroll 1
        for (int e = 0; e < 2; ++e) {
            const int w = warp + e;
            long long i = ns * w / 8;
            while (i > 0 && i < ns && __ldg(A.indices + s0 + i) == __ldg(A.indices + s0 + i - 1)) ++i;
            at[e] = i;
            cut[e] = w == 0 ? 0 : i >= ns ? nl : lower_bound(A.indices + l0, nl, __ldg(A.indices + s0 + i));
        }
        const long long sa = at[0], sn = at[1] - sa, ln = cut[1] - cut[0];
        long long D = 0, Ns = 0, Nl = 0;
        lite_exact_one<COSINE, true>(A, s0 + sa, sn, l0 + cut[0], ln, have_norms, w_idx, D, Ns, Nl);
        if ((threadIdx.x & 31) == 0) {
            s_sum[warp][0] = D;
            s_sum[warp][1] = Ns;
            s_sum[warp][2] = Nl;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            long long d = 0, nx = 0, ny = 0;
            for (int w = 0; w < 8; ++w) {
                d += s_sum[w][0];
                nx += s_sum[w][1];
                ny += s_sum[w][2];
            }
            if (have_norms) {
                nx = __ldg(A.norm2 + pr.x);
                ny = __ldg(A.norm2 + pr.y);
            }
            const double sim = lite_similarity<COSINE>(d, nx, ny, na, nb);
            A.sim[q] = sim;
            A.status[q] = sim > A.t ? BLSH_LITE_ACCEPT : BLSH_LITE_REJECT;
        }
    }
    __syncthreads();
}

template <bool COSINE>
__global__ void __launch_bounds__(256, 4) lite_exact_kernel(const LiteArgs A, const unsigned long long *heavy) {
    long long P = A.P;
    if (A.P_dev) {
        const long long pd = *A.P_dev;
        P = pd < 0 ? 0 : (pd < P ? pd : P);
    }
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    // per warp: the stage for longer rows' indices, lite_flat's area, and the
    // survivors of the current tile (offsets within it)
    extern __shared__ __align__(16) uint32_t lite_smem[];   // (read and filled 16 bytes at a time)
    uint32_t *w_idx = lite_smem + warp * kLiteWarpWords;
    uint32_t *flat = w_idx + 2 * kLiteStage;
    uint16_t *w_list = reinterpret_cast<uint16_t *>(flat + kFlatWords);
    const bool have_norms = COSINE && A.norm2 && A.scratch->norm2_valid;
    lite_heavy<COSINE>(A, heavy, have_norms, w_idx);
    if (A.scratch->work3 <= BLSH_LITE_QUEUE_CAP) return;   // every survivor was queued
    // A warp takes kLiteGrab tiles of 512 statuses per grab of the work
    // counter; a lane reads 16 statuses with one 16-byte load; the tiles'
    // survivors are listed in shared memory and computed 32 at a time, what is
    // left of a tile with the next one's.  (Not through the read-only path:
    // statuses are written in this kernel, lite_heavy's among them.)
    for (;;) {
        unsigned long long grab = 0;
        if (lane == 0) grab = atomicAdd(&A.scratch->work2, 1ull);
        grab = __shfl_sync(kFull, grab, 0);
        const long long g0 = (long long)grab * kLiteGrab * 512;
        if (g0 >= P) break;
        int listed = 0;                                    // survivors waiting, at most 31 between tiles
        for (int tt = 0; tt < kLiteGrab; ++tt) {
            const long long q0 = g0 + 512ll * tt;
            if (q0 >= P) break;
            const long long qs = q0 + 16ll * lane;
            uint32_t surv = 0;
            if (A.vec && qs + 16 <= P) {
                surv = blsh_eq16(__ldcg(reinterpret_cast<const uint4 *>(A.status + qs)), BLSH_LITE_SURVIVOR);
            } else {
                for (int i = 0; i < 16; ++i)
                    if (qs + i < P && A.status[qs + i] == BLSH_LITE_SURVIVOR) surv |= 1u << i;
            }
            const int c = __popc(surv);
            int incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += t;
            }
            const int total = __shfl_sync(kFull, incl, 31);
            if (total == 0) continue;
            __syncwarp();                                  // the previous batch's part of the list has been read
            int slot = listed + incl - c;
            for (uint32_t b = surv; b; b &= b - 1) w_list[slot++] = (uint16_t)(512 * tt + 16 * lane + __ffs(b) - 1);
            __syncwarp();
            listed += total;
            while (listed >= 32) {
                listed -= 32;
                lite_batch<COSINE>(A, g0 + w_list[listed + lane], have_norms, w_idx, flat);
            }
        }
        if (listed) lite_batch<COSINE>(A, lane < listed ? g0 + w_list[lane] : -1, have_norms, w_idx, flat);
        __syncwarp();
    }
}

// Survivors into a queue (the context's survivor queue, BLSH_LITE_QUEUE_CAP
// entries): warps scan T tiles of 512 statuses at a time in grid-stride order,
// four loads in flight, and append their survivors' indices with one atomic
// for all T.  Survivors beyond the queue are left for lite_exact_kernel.
// T = 16 where every warp has such a group: with an atomic for every
// four tiles the counter's one address (and a load in flight less often) 1e9 statuses
// took 495 us, 271 so.
template <int T>
__device__ __forceinline__ void lite_collect(const LiteArgs &A, long long P, unsigned long long *queue) {
    const int lane = threadIdx.x & 31;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long q0 = (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * (512 * T); q0 < P;
         q0 += nwarps * (512 * T)) {
        uint32_t surv[T / 2];   // two tiles' 16 bits a word
        unsigned c = 0;
#pragma unroll
        for (int t0 = 0; t0 < T; t0 += 4) {
            const long long qs = q0 + 512ll * t0 + 16ll * lane;
            uint32_t b[4] = {0u, 0u, 0u, 0u};
            if (A.vec && qs + 512 * 3 + 16 <= P) {
                uint4 v[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) v[t] = __ldg(reinterpret_cast<const uint4 *>(A.status + qs + 512 * t));
#pragma unroll
                for (int t = 0; t < 4; ++t) b[t] = blsh_eq16(v[t], BLSH_LITE_SURVIVOR);
            } else {
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    for (int i = 0; i < 16; ++i)
                        if (qs + 512 * t + i < P && A.status[qs + 512 * t + i] == BLSH_LITE_SURVIVOR) b[t] |= 1u << i;
            }
            surv[t0 / 2] = b[0] | b[1] << 16;
            surv[t0 / 2 + 1] = b[2] | b[3] << 16;
            c += __popc(surv[t0 / 2]) + __popc(surv[t0 / 2 + 1]);
        }
        unsigned incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned v = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += v;
        }
        const unsigned total = __shfl_sync(kFull, incl, 31);
        if (total == 0) continue;
        unsigned long long base = 0;
        if (lane == 31) base = atomicAdd(&A.scratch->work3, (unsigned long long)total);
        base = __shfl_sync(kFull, base, 31);
        if (base >= BLSH_LITE_QUEUE_CAP) continue;
        unsigned long long slot = base + incl - c;
#pragma unroll
        for (int t = 0; t < T / 2; ++t) {
            const long long qs = q0 + 1024ll * t + 16ll * lane;
            for (uint32_t b = surv[t]; b; b &= b - 1, ++slot) {
                const int i = __ffs(b) - 1;
                if (slot < BLSH_LITE_QUEUE_CAP) queue[slot] = (unsigned long long)(qs + (i & 15) + 512 * (i >> 4));
            }
        }
    }
}

__global__ void __launch_bounds__(256) lite_collect_kernel(const LiteArgs A, unsigned long long *queue) {
    long long P = A.P;
    if (A.P_dev) {
        const long long pd = *A.P_dev;
        P = pd < 0 ? 0 : (pd < P ? pd : P);
    }
    if (P >= 8192ll * ((long long)gridDim.x * blockDim.x >> 5)) lite_collect<16>(A, P, queue);
    else lite_collect<4>(A, P, queue);
}

// The queued survivors, a batch per warp at a time from a counter: the
// survivors of one dense tile (a bucket of near-duplicates) spread over many
// warps, and a warp with long rows takes fewer batches.
template <bool COSINE>
__global__ void __launch_bounds__(256, 4) lite_queue_kernel(const LiteArgs A, const unsigned long long *queue,
                                                            unsigned long long *heavy) {
    const unsigned long long total = A.scratch->work3;
    const unsigned long long n = total < BLSH_LITE_QUEUE_CAP ? total : BLSH_LITE_QUEUE_CAP;
    extern __shared__ __align__(16) uint32_t lite_smem[];   // (read and filled 16 bytes at a time)
    const int lane = threadIdx.x & 31;
    uint32_t *w_idx = lite_smem + (threadIdx.x >> 5) * kLiteWarpWords;
    uint32_t *flat = w_idx + 2 * kLiteStage;
    const bool have_norms = COSINE && A.norm2 && A.scratch->norm2_valid;
    // bs consecutive queue entries per warp at a time (one per lane): 32, or
    // fewer when the survivors are too few to give every warp a full batch
    // (a warp computes its batch's survivors one after the other)
    const unsigned long long nwarps = ((unsigned long long)gridDim.x * blockDim.x) >> 5;
    unsigned long long bs = (n + nwarps - 1) / nwarps;
    bs = bs < 1 ? 1 : (bs > 32 ? 32 : bs);
    for (;;) {
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(&A.scratch->work, bs);
        base = __shfl_sync(kFull, base, 0);
        if (base >= n) break;
        const long long q = lane < bs && base + lane < n ? (long long)queue[base + lane] : -1;
        lite_batch<COSINE>(A, q, have_norms, w_idx, flat, heavy);
    }
}

int lite_exact_pass(blsh_ctx *ctx, const uint2 *pairs, int64_t P, const long long *P_dev, int64_t N,
                    const int64_t *indptr, const uint32_t *indices, const float *values, double t, uint8_t *status,
                    double *sim, cudaStream_t s);

}  // namespace

extern "C" int blsh_verify_lite(blsh_ctx *ctx, const blsh_tables *tab, const uint32_t *pairs, int64_t P,
                                const int64_t *P_dev, const uint32_t *sig, int64_t N, int32_t sig_words,
                                const int64_t *indptr, const uint32_t *indices, const float *values,
                                uint8_t *status, uint16_t *n_used, double *sim, void *stream) {
    if (!ctx || !tab) return BLSH_EINVAL;
    const blsh_params &p = tab->p;
    if (tab->device != ctx->device) return blsh_fail(ctx, BLSH_EINVAL, "tables built on another device");
    if (p.h <= 0) return blsh_fail(ctx, BLSH_EINVAL, "the tables were built with h = 0");
    if (!sig || !indptr || (P > 0 && (!pairs || !status || !sim || !indices)))
        return blsh_fail(ctx, BLSH_EINVAL, "pairs, sig, status, sim, indptr and indices are required");
    if ((p.kind == BLSH_COSINE) != (values != nullptr))
        return blsh_fail(ctx, BLSH_EINVAL, "values must be given for cosine rows and only for them");
    if (P < 0 || N < 0 || N > (1ll << 32)) return blsh_fail(ctx, BLSH_EINVAL, "bad P or N");
    const int need = p.kind == BLSH_JACCARD ? p.h : (p.h + 31) / 32;
    if (sig_words < need || sig_words % 4)
        return blsh_fail(ctx, BLSH_EINVAL, "sig_words must be a multiple of 4 covering h hashes");
    if (!blsh_aligned(sig, 16) || !blsh_aligned(pairs, 8) || !blsh_aligned(sim, 8) || !blsh_aligned(indptr, 8) ||
        !blsh_aligned(n_used, 2) || !blsh_aligned(P_dev, 8))
        return blsh_fail(ctx, BLSH_EINVAL, "misaligned pointer");
    blsh_device_guard g(ctx->device);
    cudaStream_t s = blsh_stream(stream);
    VerifyArgs A;
    A.pairs = reinterpret_cast<const uint2 *>(pairs);
    A.P = P;
    A.P_dev = reinterpret_cast<const long long *>(P_dev);
    A.sig = sig;
    A.N = N;
    A.W = sig_words;
    A.k = p.k;
    A.chunk_words = p.kind == BLSH_JACCARD ? p.k : p.k / 32;
    A.levels = p.h / p.k;
    A.lite = 1;
    A.conc_words = tab->conc_words;
    A.est_stride = p.n_max + 1;
    A.min_matches = tab->min_matches;
    A.conc_bits = tab->conc_bits;
    A.conc_lo = tab->conc_lo;
    A.conc_upper = tab->conc_upper ? 1 : 0;
    A.est_tab = tab->est;
    A.status = status;
    A.n_used = n_used;
    A.m_out = nullptr;
    A.est_out = nullptr;
    A.sim_out = sim;
    A.stop_hist = nullptr;
    A.scratch = ctx->scratch;
    A.lite_levels = 0;
    A.lstatus = nullptr;
    A.ln_used = nullptr;
    A.lsim = nullptr;
    A.cap_levels = A.levels;
    A.need = nullptr;
    const blsh_plan plan = blsh_plan_for(ctx, tab, P, blsh_packed_outputs(pairs, status, n_used, nullptr, nullptr, nullptr));
    A.grab = (plan.grab + 31) / 32 * 32;
    int rc = blsh_launch_verify(ctx, A, plan, s);
    if (rc) return rc;
    if (P == 0) return BLSH_OK;
    return lite_exact_pass(ctx, A.pairs, P, A.P_dev, N, indptr, indices, values, p.t, status, sim, s);
}

namespace {

// Pass 2 of Algorithm 2: the exact similarity of every survivor.
int lite_exact_pass(blsh_ctx *ctx, const uint2 *pairs, int64_t P, const long long *P_dev, int64_t N,
                    const int64_t *indptr, const uint32_t *indices, const float *values, double t, uint8_t *status,
                    double *sim, cudaStream_t s) {
    LiteArgs L;
    L.pairs = pairs;
    L.P = P;
    L.P_dev = P_dev;
    L.indptr = indptr;
    L.indices = indices;
    L.values = values;
    L.t = t;
    L.status = status;
    L.sim = sim;
    L.scratch = ctx->scratch;
    L.vec = blsh_aligned(status, 16);
    L.N = N;
    L.norm2 = nullptr;
    // the rows' squared norms once per call, in the buffer blsh_ctx_reserve
    // allocated; with more rows than were reserved each survivor forms its
    // two sums itself (no allocation here: this is a hot call)
    if (values && N > 0 && ctx->norm2_cap >= N) L.norm2 = (const long long *)ctx->norm2;
    // survivors: queued (balanced over warps), then any beyond the queue in place
    // work, work2, work3, recheck_count (survivors of two long rows) .. hash_work (the next of them)
    BLSH_CUDA(ctx, cudaMemsetAsync(&ctx->scratch->work, 0, offsetof(blsh_dev_scratch, norm2_valid) -
                                                              offsetof(blsh_dev_scratch, work), s));
    unsigned long long *queue = ctx->lite_queue;
    unsigned long long *heavy = reinterpret_cast<unsigned long long *>(ctx->recheck_queue);   // [BLSH_RECHECK_CAP]
    blsh_time_start(ctx, s);
    lite_collect_kernel<<<ctx->sm_count * 8, 256, 0, s>>>(L, queue);
    BLSH_LAUNCHED(ctx, "lite_collect_kernel");
    if (L.norm2) {
        const long long blocks = (N + 31) / 32, cap = (long long)ctx->sm_count * 32;   // 32 rows a CTA
        blsh_time_start(ctx, s);
        row_norm2_kernel<<<(unsigned)(blocks < cap ? blocks : cap), 256, 0, s>>>(
            indptr, values, N, const_cast<long long *>(L.norm2), ctx->scratch);
        BLSH_LAUNCHED(ctx, "row_norm2_kernel");
    }
    // (four CTAs an SM: their launch bounds' registers, and 55 KB of shared memory)
    const size_t smem = 8 * kLiteWarpWords * sizeof(uint32_t);
    const unsigned grid = 4u * ctx->sm_count;
    auto run = [&](auto queue_kernel, auto exact_kernel) -> int {
        BLSH_CUDA(ctx, cudaFuncSetAttribute(queue_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        BLSH_CUDA(ctx, cudaFuncSetAttribute(exact_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        blsh_time_start(ctx, s);
        queue_kernel<<<grid, 256, smem, s>>>(L, queue, heavy);
        BLSH_LAUNCHED(ctx, "lite_queue_kernel");
        blsh_time_start(ctx, s);
        exact_kernel<<<grid, 256, smem, s>>>(L, heavy);
        BLSH_LAUNCHED(ctx, "lite_exact_kernel");
        return BLSH_OK;
    };
    return values ? run(lite_queue_kernel<true>, lite_exact_kernel<true>)
                  : run(lite_queue_kernel<false>, lite_exact_kernel<false>);
}

}  // namespace

namespace {

int verify_both(blsh_ctx *ctx, const blsh_tables *tab, int32_t hash_limit, const uint32_t *pairs, int64_t P,
                const int64_t *P_dev, const uint32_t *sig, int64_t N, int32_t sig_words, uint8_t *status,
                uint16_t *n_used, uint16_t *m, float *est, uint64_t *stop_hist, const int64_t *indptr,
                const uint32_t *indices, const float *values, uint8_t *lite_status, uint16_t *lite_n_used,
                double *sim, uint8_t *need, void *stream) {
    if (!ctx || !tab) return BLSH_EINVAL;
    const blsh_params &p = tab->p;
    if (tab->device != ctx->device) return blsh_fail(ctx, BLSH_EINVAL, "tables built on another device");
    if (p.h <= 0) return blsh_fail(ctx, BLSH_EINVAL, "the tables were built with h = 0");
    if (hash_limit % p.k || hash_limit < p.h || hash_limit > p.n_max)
        return blsh_fail(ctx, BLSH_EINVAL, "hash_limit must be a multiple of k in [h, n_max]");
    if (hash_limit < p.n_max && !need) return blsh_fail(ctx, BLSH_EINVAL, "need is required below n_max");
    if (!indptr || (P > 0 && (!lite_status || !sim || !indices)))
        return blsh_fail(ctx, BLSH_EINVAL, "lite_status, sim, indptr and indices are required");
    if ((p.kind == BLSH_COSINE) != (values != nullptr))
        return blsh_fail(ctx, BLSH_EINVAL, "values must be given for cosine rows and only for them");
    if (!blsh_aligned(sim, 8) || !blsh_aligned(indptr, 8) || !blsh_aligned(lite_n_used, 2))
        return blsh_fail(ctx, BLSH_EINVAL, "misaligned pointer");
    VerifyArgs A;
    int rc = blsh_make_verify_args(ctx, tab, pairs, P, P_dev, sig, N, sig_words, status, n_used, m, est,
                                   stop_hist, A);
    if (rc) return rc;
    A.lite_levels = p.h / p.k;
    A.lstatus = lite_status;
    A.ln_used = lite_n_used;
    A.lsim = sim;
    A.cap_levels = hash_limit / p.k;
    A.need = need;
    const blsh_plan plan =
        blsh_plan_for(ctx, tab, P, blsh_packed_outputs(pairs, status, n_used, m, lite_status, lite_n_used));
    A.grab = (plan.grab + 31) / 32 * 32;
    blsh_device_guard g(ctx->device);
    cudaStream_t s = blsh_stream(stream);
    if (stop_hist) BLSH_CUDA(ctx, cudaMemsetAsync(stop_hist, 0, sizeof(uint64_t) * tab->levels, s));
    rc = blsh_launch_verify(ctx, A, plan, s);
    if (rc) return rc;
    if (P == 0) return BLSH_OK;
    return lite_exact_pass(ctx, A.pairs, P, A.P_dev, N, indptr, indices, values, p.t, lite_status, sim, s);
}

}  // namespace

extern "C" int blsh_verify_both(blsh_ctx *ctx, const blsh_tables *tab, const uint32_t *pairs, int64_t P,
                                const int64_t *P_dev, const uint32_t *sig, int64_t N, int32_t sig_words,
                                uint8_t *status, uint16_t *n_used, uint16_t *m, float *est, uint64_t *stop_hist,
                                const int64_t *indptr, const uint32_t *indices, const float *values,
                                uint8_t *lite_status, uint16_t *lite_n_used, double *sim, void *stream) {
    if (!ctx || !tab) return BLSH_EINVAL;
    return verify_both(ctx, tab, tab->p.n_max, pairs, P, P_dev, sig, N, sig_words, status, n_used, m, est,
                       stop_hist, indptr, indices, values, lite_status, lite_n_used, sim, nullptr, stream);
}

extern "C" int blsh_verify_both_capped(blsh_ctx *ctx, const blsh_tables *tab, int32_t hash_limit,
                                       const uint32_t *pairs, int64_t P, const int64_t *P_dev, const uint32_t *sig,
                                       int64_t N, int32_t sig_words, uint8_t *status, uint16_t *n_used, uint16_t *m,
                                       float *est, uint64_t *stop_hist, const int64_t *indptr,
                                       const uint32_t *indices, const float *values, uint8_t *lite_status,
                                       uint16_t *lite_n_used, double *sim, uint8_t *need, void *stream) {
    return verify_both(ctx, tab, hash_limit, pairs, P, P_dev, sig, N, sig_words, status, n_used, m, est, stop_hist,
                       indptr, indices, values, lite_status, lite_n_used, sim, need, stream);
}
