// srp_dense.cu -- sign random projections of dense rows (Section 4.2, "LSH
// family"): bit j of row i = [x_i . r_j >= 0].
//
// Tensor-core path (bits a multiple of 256, any d up to 4096: K is padded with
// zeros to Kpad, the next multiple of 64):
//   1. srp_dense_prep: X and R become BF16 pairs hi + lo with
//      hi = bf16(v), lo = bf16(v - hi) (|v - hi - lo| <= 2^-16 |v|), written in
//      the tile layout the tensor cores read (128- and 256-row tiles of 64
//      K-values, 128-byte rows, 16-byte chunks XOR-swizzled by row), plus the
//      L2 norms of the rows of X and the columns of R.
//   2. srp_dense_tc_persistent: one CTA per SM walks tiles of 128 rows x 256
//      bits; the K dimension streams through a two-stage shared-memory ring
//      filled by bulk copies (cp.async.bulk, completion on mbarriers); one
//      thread issues tcgen05.mma (BF16 x BF16 -> FP32 in tensor memory) for
//      hi*hi, hi*lo and lo*hi into one of two accumulators; four epilogue
//      warps read the other accumulator back (tcgen05.ld) and set a bit
//      wherever |p| > margin * |x_i| * |r_j|, marking every other sign in a
//      bit map.
//   3. srp_dense_recheck_kernel: each marked sign is recomputed in FP32 with a
//      rigorous error bound, then in FP64 with one, and, if neither can decide
//      it, as the FP64 sum over coordinates 0..d-1 in order -- the oracle's
//      definition -- so every bit is exact whenever the margin bounds the
//      tensor-core error.
// The error of step 2 is at most 3.1 * 2^-16 sum|x_i r_ij| from the split
// plus the FP32 accumulation of 3 Kpad products; the rigorous margin used when
// the caller passes margin <= 0 is (2^-14 + 3 Kpad 2^-22) * 1.25, applied to
// |x| |r| >= sum|x_i r_ij|.  That the accumulation errs by less than 2^-22 a
// product is taken from measurement, not from a document: over widths of 1 to
// 4,096 and Gaussian, one-signed, widely spread and outlying values the
// accumulators differ from the FP64 products by at most 0.20 of the margin (one
// coordinate: 2.7e-5 of 1.34e-4, the split), 0.06 at 64, 0.01 from 300 on (4,096
// one-signed ones: 1.9e-5 of 3.7e-3), and every sign is that of the FP64 sum.
//
// A width that is no multiple of 64 takes the same path since the padding
// costs at most one K stage, while the CUDA cores need 2 d operations a sign
// at 1/50 of the tensor rate: 99,991 x 300 x 1,024 bits took 36.4 ms on the
// CUDA cores' kernel of that time, 289 us here.
//
// Every other shape uses srp_dense_simt_kernel (hashing.cu): FP32 sums with
// the same kind of bound and an FP64 recheck.
#include <cuda_bf16.h>
#include <math.h>

#include <atomic>

#include "common.cuh"

int blsh_srp_dense_simt(blsh_ctx *ctx, const float *X, int64_t N, int32_t d, const float *R, int32_t bits,
                        uint32_t *sig, cudaStream_t s);

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int BM = 128;                   // rows of X per CTA
constexpr int BN = 256;                   // bits per CTA
constexpr int BK = 64;                    // K values per stage (128 bytes of BF16 per row)
constexpr int TILE_A = BM * BK * 2;       // 16 KiB
constexpr int TILE_B = BN * BK * 2;       // 32 KiB
constexpr int STAGE_BYTES = 2 * TILE_A + 2 * TILE_B;   // hi and lo of both operands: 96 KiB
constexpr int STAGES = 2;
constexpr long long kWaitPolls = 1ll << 24;

// byte offset of element k (0..63) of row r inside a 128-byte-row tile with
// the 128-byte swizzle: 16-byte chunk c = k/8 is stored at chunk c ^ (r % 8)
__host__ __device__ inline int swz_offset(int r, int k) { return r * 128 + ((((k >> 3) ^ (r & 7))) << 4) + (k & 7) * 2; }

__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

// ---- preparation --------------------------------------------------------------

// One launch prepares both operands: the first r_blocks CTAs take 32 columns of R each, the others the rows of X.
//
// R: a CTA walks K in stages of 64: a 64 x 32 tile is read in 128-byte rows,
// turned in shared memory, and each thread writes eight K values of a column
// (16 bytes of the hi and lo operands, which are N-major rows of K values, and
// 32 bytes of Rt, FP32 R transposed, read by the rechecks).  One thread per
// column, with its 2-byte stores 128 bytes apart, had taken 133 us at
// 384 x 1,024 (of a 169 us call for 1,000 rows) and 102 us at 256 x 1,024;
// this form takes 11 us, both operands together, for those 1,000 rows.
// X: one warp per row (rows >= N are zero-filled up to the padded tile), four
// consecutive values a lane at a time (VEC: d a multiple of 4, so that every
// row starts on 16 bytes).
// xnorm, rnorm: |x_i|, |r_j| in FP32 rounded up, infinity outside
// [1e-30, 1e18] (norm_or_inf), where an infinite bound sends every sign to the
// recheck.  Up to 1e18 no partial sum of the tensor cores can overflow (each is
// at most |x_i| |r_j| <= 1e36); down to 1e-30 what an operand's split loses to
// underflow is below 2^-20 of its norm.  A product's underflow stays far below
// margin |x_i| |r_j| while |x_i| |r_j| >= 1e-30 (margin >= 3e-4: 3e-34), which
// the epilogue asks of a row and the smallest column.
constexpr int kPrepCols = 32;
__device__ __forceinline__ float norm_or_inf(float ss) {
    const float n = __fsqrt_ru(ss) * 1.0001f;   // (ss: squares added upwards, so never too small)
    return n >= 1e-30f && n <= 1e18f ? n : INFINITY;
}

template <bool VEC>
__global__ void __launch_bounds__(256) srp_dense_prep(
    const float *__restrict__ X, long long N, long long Npad, int d, int KT, unsigned char *__restrict__ Xh,
    unsigned char *__restrict__ Xl, float *__restrict__ xnorm, const float *__restrict__ R, int bits,
    unsigned char *__restrict__ Rh, unsigned char *__restrict__ Rl, float *__restrict__ rnorm,
    float *__restrict__ Rt, int r_blocks) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if ((int)blockIdx.x < r_blocks) {
        __shared__ float tile[BK][kPrepCols + 1];
        const int j0 = blockIdx.x * kPrepCols;
        const int c = threadIdx.x >> 3, q = threadIdx.x & 7;   // this thread's column and 16-byte chunk
        const int j = j0 + c;
        const int nt = j / BN, jj = j % BN;
        float ss = 0.0f;
        for (int kt = 0; kt < KT; ++kt) {
#pragma unroll
            for (int i = 0; i < BK / 8; ++i) {
                const int kk = warp + 8 * i, k = kt * BK + kk;
                tile[kk][lane] = k < d ? __ldg(R + (size_t)k * bits + j0 + lane) : 0.0f;
            }
            __syncthreads();
            __align__(16) __nv_bfloat16 hi[8], lo[8];
            __align__(16) float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                v[i] = tile[8 * q + i][c];
                hi[i] = __float2bfloat16_rn(v[i]);
                lo[i] = __float2bfloat16_rn(v[i] - __bfloat162float(hi[i]));
                ss = __fmaf_ru(v[i], v[i], ss);
            }
            const size_t off = ((size_t)nt * KT + kt) * TILE_B + swz_offset(jj, 8 * q);
            *reinterpret_cast<uint4 *>(Rh + off) = *reinterpret_cast<const uint4 *>(hi);
            *reinterpret_cast<uint4 *>(Rl + off) = *reinterpret_cast<const uint4 *>(lo);
            float4 *t = reinterpret_cast<float4 *>(Rt + (size_t)j * (KT * BK) + kt * BK + 8 * q);
            t[0] = make_float4(v[0], v[1], v[2], v[3]);
            t[1] = make_float4(v[4], v[5], v[6], v[7]);
            __syncthreads();
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) ss = __fadd_ru(ss, __shfl_xor_sync(kFull, ss, o));
        if (q == 0) rnorm[j] = norm_or_inf(ss);
        return;
    }
    const long long warps = (long long)(gridDim.x - r_blocks) * (blockDim.x >> 5);
    for (long long r = (long long)(blockIdx.x - r_blocks) * (blockDim.x >> 5) + warp; r < Npad; r += warps) {
        const long long mt = r / BM;
        const int rr = (int)(r % BM);
        float ss = 0.0f;
        for (int k0 = 4 * lane; k0 < KT * BK; k0 += 128) {
            float a[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            if (r < N) {
                if (VEC) {
                    if (k0 < d) {
                        const float4 v = __ldg(reinterpret_cast<const float4 *>(X + (size_t)r * d + k0));
                        a[0] = v.x; a[1] = v.y; a[2] = v.z; a[3] = v.w;
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (k0 + i < d) a[i] = __ldg(X + (size_t)r * d + k0 + i);
                }
            }
            __align__(8) __nv_bfloat16 hi[4], lo[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                hi[i] = __float2bfloat16_rn(a[i]);
                lo[i] = __float2bfloat16_rn(a[i] - __bfloat162float(hi[i]));
                ss = __fmaf_ru(a[i], a[i], ss);
            }
            const int kt = k0 / BK, kk = k0 % BK;
            const size_t tile = ((size_t)mt * KT + kt) * TILE_A;
            *reinterpret_cast<uint2 *>(Xh + tile + swz_offset(rr, kk)) = *reinterpret_cast<const uint2 *>(hi);
            *reinterpret_cast<uint2 *>(Xl + tile + swz_offset(rr, kk)) = *reinterpret_cast<const uint2 *>(lo);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ss = __fadd_ru(ss, __shfl_xor_sync(kFull, ss, o));
        if (lane == 0) xnorm[r] = norm_or_inf(ss);
    }
}

// ---- tcgen05 / mbarrier / bulk-copy helpers ------------------------------------

__device__ __forceinline__ void mbar_init(unsigned long long *bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long *bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long *bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait: false if the phase did not complete within kWaitPolls polls
__device__ __forceinline__ bool mbar_wait(unsigned long long *bar, unsigned parity) {
    for (long long i = 0; i < kWaitPolls; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, unsigned bytes, unsigned long long *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows
// 128 bytes apart, 8-row groups 1024 bytes apart.
__device__ __forceinline__ unsigned long long smem_desc(const void *p) {
    const unsigned long long addr = smem_u32(p);
    unsigned long long d = 0;
    d |= (addr & 0x3FFFFull) >> 4;          // start address
    d |= 1ull << 16;                         // leading-dimension byte offset (unused for this layout)
    d |= (1024ull >> 4) << 32;               // stride-dimension byte offset
    d |= 1ull << 46;                         // descriptor version
    d |= 2ull << 61;                         // 128-byte swizzle
    return d;
}

// Instruction descriptor: BF16 x BF16 -> FP32, both operands K-major, M = 128, N = 256.
constexpr unsigned kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(BN >> 3) << 17) | ((unsigned)(BM >> 4) << 24);

__device__ __forceinline__ void mma_bf16(unsigned tmem_d, unsigned long long a, unsigned long long b, unsigned acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(kIdesc), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void mma_commit(unsigned long long *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }

// 32 consecutive FP32 columns of this warp's 32 TMEM lanes
__device__ __forceinline__ void tmem_ld32(unsigned taddr, float (&v)[32]) {
    unsigned r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// ---- the persistent, warp-specialised tensor-core kernel -------------------------
//
// One CTA per SM walks the tiles t = blockIdx.x, blockIdx.x + gridDim.x, ...
// (tile t: rows 128 (t / tiles_n), bits 256 (t % tiles_n), so consecutive
// tiles of a CTA share their rows of X).  Six warps:
//   warp 0  producer: bulk copies of each K stage into the two-stage ring;
//   warp 1  MMA issuer (one thread): 12 tcgen05.mma per K stage into one of
//           two 256-column accumulators in tensor memory (512 columns), so
//           the epilogue of one tile runs while the next tile accumulates;
//   warps 2-9 epilogue: warp w reads TMEM lanes 32 (w % 4) .. +31 (rows of
//           the tile) in columns 128 ((w - 2) / 4) .. +127, tests each value
//           against margin |x_i| |r_j| (margin |r_j| staged in shared memory
//           for all bits), writes the decided bits and marks the others.
// Barriers: full/empty per ring stage (bulk-copy bytes / MMA commit), and
// acc_full/acc_empty per accumulator (MMA commit / 128 epilogue arrivals).
// Every wait is bounded; a role that gives up records the failure and
// stops, and the others give up in turn.
constexpr int kEpiWarps = 8;   // two per TMEM lane quarter, each taking half of a tile's 256 columns
constexpr int kTcThreads = 32 * (2 + kEpiWarps);

__device__ __forceinline__ void mbar_arrive(unsigned long long *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__global__ void __launch_bounds__(kTcThreads, 1) srp_dense_tc_persistent(
    const unsigned char *__restrict__ Xh, const unsigned char *__restrict__ Xl, const unsigned char *__restrict__ Rh,
    const unsigned char *__restrict__ Rl, const float *__restrict__ xnorm, const float *__restrict__ rnorm,
    long long N, int d, int bits, float margin, uint32_t *__restrict__ sig, uint32_t *__restrict__ und,
    long long tiles_total, blsh_dev_scratch *scratch) {
    extern __shared__ __align__(1024) unsigned char dyn_smem[];
    unsigned char *ring = reinterpret_cast<unsigned char *>(((uintptr_t)dyn_smem + 1023) & ~(uintptr_t)1023);
    float *s_mr = reinterpret_cast<float *>(ring + (size_t)STAGES * STAGE_BYTES);   // [bits]: margin |r_j|
    for (int j = threadIdx.x; j < bits; j += blockDim.x) s_mr[j] = margin * __ldg(rnorm + j);
    __shared__ __align__(8) unsigned long long full_bar[STAGES], empty_bar[STAGES], acc_full[2], acc_empty[2];
    __shared__ __align__(8) unsigned long long mma_done;
    __shared__ unsigned tmem_base;
    __shared__ volatile int s_fail;
    const int KT = (d + BK - 1) / BK;
    const int tiles_n = bits / BN;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(2 * BN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int st = 0; st < STAGES; ++st) {
            mbar_init(&full_bar[st], 1);
            mbar_init(&empty_bar[st], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 32 * kEpiWarps);
        }
        mbar_init(&mma_done, 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const unsigned tmem = tmem_base;

    if (warp == 0) {
        if (lane == 0) {   // producer
            long long it = 0;
            for (long long t = blockIdx.x; t < tiles_total && !s_fail; t += gridDim.x) {
                const long long mt = t / tiles_n;
                const int nt = (int)(t % tiles_n);
                for (int kb = 0; kb < KT; ++kb, ++it) {
                    const int st = (int)(it % STAGES);
                    const unsigned use = (unsigned)(it / STAGES);
                    if (!mbar_wait(&empty_bar[st], (use & 1u) ^ 1u)) {   // the MMAs reading stage st are done
                        s_fail = 1;
                        break;
                    }
                    unsigned char *sp = ring + (size_t)st * STAGE_BYTES;
                    const size_t ta = ((size_t)mt * KT + kb) * TILE_A, tb = ((size_t)nt * KT + kb) * TILE_B;
                    mbar_expect_tx(&full_bar[st], STAGE_BYTES);
                    bulk_g2s(sp, Xh + ta, TILE_A, &full_bar[st]);
                    bulk_g2s(sp + TILE_A, Xl + ta, TILE_A, &full_bar[st]);
                    bulk_g2s(sp + 2 * TILE_A, Rh + tb, TILE_B, &full_bar[st]);
                    bulk_g2s(sp + 2 * TILE_A + TILE_B, Rl + tb, TILE_B, &full_bar[st]);
                }
            }
            // the last copy into each stage has landed before the CTA ends
            // (at once when its MMAs consumed it; a bounded wait otherwise)
            for (int st = 0; st < STAGES; ++st)
                if (it > st) mbar_wait(&full_bar[st], (unsigned)(((it - 1 - st) / STAGES) & 1));
        }
    } else if (warp == 1) {
        if (lane == 0) {   // MMA issuer
            long long it = 0, tc = 0;
            for (long long t = blockIdx.x; t < tiles_total && !s_fail; t += gridDim.x, ++tc) {
                const int buf = (int)(tc & 1);
                const unsigned use_acc = (unsigned)(tc >> 1);
                if (!mbar_wait(&acc_empty[buf], (use_acc & 1u) ^ 1u)) {   // the epilogue is done with it
                    s_fail = 1;
                    break;
                }
                fence_after();
                const unsigned acc = tmem + (unsigned)(buf * BN);
                bool ok = true;
                for (int kb = 0; kb < KT; ++kb, ++it) {
                    const int st = (int)(it % STAGES);
                    const unsigned use = (unsigned)(it / STAGES);
                    if (!mbar_wait(&full_bar[st], use & 1u)) {
                        ok = false;
                        break;
                    }
                    fence_after();
                    unsigned char *sp = ring + (size_t)st * STAGE_BYTES;
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk) {   // K = 16 per MMA: 32 bytes along the 128-byte row
                        const unsigned long long ah = smem_desc(sp + kk * 32), al = smem_desc(sp + TILE_A + kk * 32);
                        const unsigned long long bh = smem_desc(sp + 2 * TILE_A + kk * 32);
                        const unsigned long long bl = smem_desc(sp + 2 * TILE_A + TILE_B + kk * 32);
                        mma_bf16(acc, ah, bh, (kb | kk) != 0);
                        mma_bf16(acc, ah, bl, 1u);
                        mma_bf16(acc, al, bh, 1u);
                    }
                    mma_commit(&empty_bar[st]);   // stage st is free once these MMAs finish
                }
                if (!ok) {
                    s_fail = 1;
                    break;
                }
                mma_commit(&acc_full[buf]);       // the tile's accumulator is final once all its MMAs finish
            }
            // every MMA issued has finished before tensor memory is freed
            mma_commit(&mma_done);
            mbar_wait(&mma_done, 0u);
        }
    } else {   // epilogue warps
        const int ew = warp & 3;                  // TMEM lanes 32 ew .. 32 ew + 31
        const int half = (warp - 2) >> 2;         // columns 128 half .. 128 half + 127
        const int words = bits >> 5;
        const bool sig16 = ((uintptr_t)sig & 15) == 0;
        float mr_min = INFINITY;
        for (int j = lane; j < bits; j += 32) mr_min = fminf(mr_min, s_mr[j]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mr_min = fminf(mr_min, __shfl_xor_sync(kFull, mr_min, o));
        long long tc = 0;
        for (long long t = blockIdx.x; t < tiles_total && !s_fail; t += gridDim.x, ++tc) {
            const long long mt = t / tiles_n;
            const int nt = (int)(t % tiles_n);
            const int buf = (int)(tc & 1);
            const unsigned use_acc = (unsigned)(tc >> 1);
            if (!__all_sync(kFull, mbar_wait(&acc_full[buf], use_acc & 1u))) {   // the same verdict for the warp
                s_fail = 1;
                break;
            }
            fence_after();
            const long long row = mt * BM + ew * 32 + lane;
            float xn = row < N ? __ldg(xnorm + row) : 0.0f;
            if (!(xn * mr_min >= margin * 1e-30f)) xn = INFINITY;
            uint32_t word[4], mark[4];
#pragma unroll
            for (int cc = 0; cc < 4; ++cc) {
                const int c = half * 4 + cc;
                float v[32];
                tmem_ld32(tmem + ((unsigned)(ew * 32) << 16) + (unsigned)(buf * BN + c * 32), v);
                const float *mr = s_mr + nt * BN + c * 32;
                uint32_t w = 0, u = 0;
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    w |= (uint32_t)(v[i] >= 0.0f) << i;
                    u |= (uint32_t)!(fabsf(v[i]) > xn * mr[i]) << i;   // inside the margin (or NaN): recheck
                }
                word[cc] = w & ~u;
                mark[cc] = u;
            }
            if (row < N) {
                const size_t at = (size_t)row * words + nt * (BN / 32) + half * 4;
                if (sig16) {
                    *reinterpret_cast<uint4 *>(sig + at) = make_uint4(word[0], word[1], word[2], word[3]);
                } else {
#pragma unroll
                    for (int cc = 0; cc < 4; ++cc) sig[at + cc] = word[cc];
                }
                *reinterpret_cast<uint4 *>(und + at) = make_uint4(mark[0], mark[1], mark[2], mark[3]);
            }
            // the accumulator may be overwritten now
            fence_before();
            mbar_arrive(&acc_empty[buf]);
        }
    }
    fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && s_fail) blsh_dev_error(scratch, BLSH_EDEVICE, -1, 0ull);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * BN) : "memory");
}

// The marked signs.  An item is 32 words of marks, a lane a word: 32 words of a
// row, or 16 or 8 words of two or four rows where the width asks for it.  They
// are listed in shared memory row by row, and the warp forms eight sums at a
// time: lane l takes coordinates 4 l .. 4 l + 3 of every 128 of x_i (kept in
// registers for all of the row's signs where d <= 256) and of the columns, in
// paired FMAs, and the eight sums meet in nine shuffles.  Three stages, each with a rigorous bound:
//   FP32: no term passes through more than 2 ceil(d/128) + 6 roundings, so the
//   sum errs by at most that many u |x_i| |r_j| (norms rounded up; infinite
//   where they could over- or underflow), or, if that does not decide, u sum|p|
//   of the same chains;
//   then FP64 partial sums of the exact products, a lane's coordinates l, l + 32, ...
//   (error at most (d/32 + 6) 2^-53 sum|p|: a sign it decides is the sign of
//   the exact sum and of the oracle's sum, which errs by less than d 2^-53
//   sum|p|); a sum that is not finite, or of products that are all zero, is the
//   same in every order;
//   the rest, exact ties, as the FP64 sum over coordinates 0..d-1 in order --
//   exactly the oracle's sum -- a lane each.  A zero row's sums need no FP64.
//   Three open signs or more among eight are taken for ties at once: the middle
//   stages, the warp's for every sign, cost 3 to 5 us each where a lane's sum
//   costs 2 us for 32 of them (100 x 64 x 256 bits of +-1, a tenth ties: 846 us,
//   75 here).
//
// What bounds it: the reads of the columns, 4 d bytes a sign, from L2 and L1.
// A queue of (row, bit) entries, eight lanes each, read x_i as well for every
// sign: 2,077 us for the 1.3e7 signs that 1e6 x 256 x 1,024 bits leave inside
// the margin 1e-3, and the queue's appends cost the tensor-core kernel 200 us
// (1,049 us, with marks 840 us); where most signs were ties it overflowed and
// the epilogue summed them itself (1e5 x 256, 1% of them zero: 51 ms, now 0.23 ms).
// Here x_i is read once, and the sums take 1,090 us (13 TB/s of columns).
// Items of 8 words of 4 rows, so that an SM's L1 holds its part of the columns,
// take 1,695 us: a row's few signs no longer fill a batch.  24 warps of 80
// registers: with 32 of 64 1,230 us, with 28 1,263 us, with 20 1,137 us; four
// sums at a time instead of eight 1,311 us.
constexpr int kReWarps = 24;
constexpr int kReList = 512;   // signs listed at a time

struct RecheckArgs {
    const uint32_t *und;
    const float *X, *Rt, *xnorm, *rnorm;
    long long N;
    int d, ldr, bits;
    int part_words;   // words of a row an item covers: 8, 16 or 32
    uint32_t *sig;
    blsh_dev_scratch *scratch;
};

// coordinates c .. c + 3 of x (zeros past d), as two pairs (CG: not kept in L1)
template <bool VEC, bool CG>
__device__ __forceinline__ ulonglong2 x_pairs(const float *__restrict__ x, int c, int d) {
    ulonglong2 v = make_ulonglong2(0ull, 0ull);
    if (VEC) {
        if (c < d) v = CG ? __ldcg(reinterpret_cast<const ulonglong2 *>(x + c)) : __ldg(reinterpret_cast<const ulonglong2 *>(x + c));
    } else {
        float a[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = c + i >= d ? 0.0f : CG ? __ldcg(x + c + i) : __ldg(x + c + i);
        v = make_ulonglong2(f2_pack(a[0], a[1]), f2_pack(a[2], a[3]));
    }
    return v;
}

// The warp's sign of x . r where the norms did not decide it: +1, -1, or 0 for
// a tie (the ordered sum is needed).  zero: the exact sum is zero.
template <bool VEC>
__device__ __noinline__ int sign_by_magnitude(const float *__restrict__ x, const float *__restrict__ r, int d, int ldr,
                                              float acc, float roundings, bool *zero) {
    const int lane = threadIdx.x & 31;
    unsigned long long m2 = 0ull;
    for (int c = 4 * lane; c < ldr; c += 128) {
        const ulonglong2 u = x_pairs<VEC, false>(x, c, d), v = __ldg(reinterpret_cast<const ulonglong2 *>(r + c));
        constexpr unsigned long long kAbs = 0x7fffffff7fffffffull;
        m2 = f2_fma(u.x & kAbs, v.x & kAbs, m2);
        m2 = f2_fma(u.y & kAbs, v.y & kAbs, m2);
    }
    float m0, m1;
    f2_unpack(m2, m0, m1);
    float mag = m0 + m1;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mag += __shfl_xor_sync(kFull, mag, o);
    if (fabsf(acc) > 1.25f * roundings * 5.9604644775390625e-8f * mag + (float)(d + 8) * 1.4e-45f)
        return acc > 0.0f ? 1 : -1;
    double p = 0.0, q = 0.0;
    for (int c = lane; c < d; c += 32) {
        const double t = (double)__ldg(x + c) * (double)__ldg(r + c);
        p += t;
        q += fabs(t);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        p += __shfl_xor_sync(kFull, p, o);
        q += __shfl_xor_sync(kFull, q, o);
    }
    *zero = q == 0.0;
    if (!(fabs(p) <= 1.7976931348623157e308) || q == 0.0) return p >= 0.0 ? 1 : -1;   // NaN: no bit
    if (fabs(p) > 1.25 * (double)(d + 8) * 1.1102230246251565e-16 * q + (double)(d + 8) * 5e-324)
        return p > 0.0 ? 1 : -1;
    return 0;
}

template <bool VEC, bool REG>
__global__ void __launch_bounds__(32 * kReWarps, 1) srp_dense_recheck_kernel(const RecheckArgs A) {
    __shared__ __align__(16) uint16_t s_list[kReWarps][kReList + 8];   // columns within the part, padded to eight
    __shared__ uint32_t s_bits[kReWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int W = A.part_words, rows = 32 / W, words = A.bits >> 5, parts = words / W, d = A.d, ldr = A.ldr;
    const int part = blockIdx.x % parts;
    const long long groups = (A.N + rows - 1) / rows;
    const long long stride = (long long)(gridDim.x / parts) * kReWarps;
    const float *__restrict__ Rt = A.Rt + (size_t)part * W * 32 * ldr;
    const float *__restrict__ rn = A.rnorm + part * W * 32;
    const unsigned ldr4 = 4u * ldr;
    // this lane's coordinates of a column (those past its end: x is zero there)
    const char *r0 = reinterpret_cast<const char *>(Rt + (4 * lane < ldr ? 4 * lane : 0));
    const char *r1 = reinterpret_cast<const char *>(Rt + (128 + 4 * lane < ldr ? 128 + 4 * lane : 0));
    const float roundings = (float)(2 * ((d + 127) / 128) + 6);
    const float tiny = (float)(d + 8) * 1.4e-45f;
    constexpr unsigned long long kAbs = 0x7fffffff7fffffffull;
    uint16_t *list = s_list[warp];
    uint32_t *bits = s_bits[warp];
    unsigned long long done = 0;
    unsigned zeros = 0;
    const int wrow = lane / W, wword = part * W + lane % W;
    auto marks = [&](long long g) -> uint32_t {
        const long long row = g * rows + wrow;
        return g < groups && row < A.N ? __ldcs(A.und + (size_t)row * words + wword) : 0u;
    };
    // no more items than warps: in as many CTAs as can be; else a CTA's follow
    // each other (spread over the CTAs 1e5 x 300 x 1,024 bits took 137 us, 131 so)
    const long long ctas = gridDim.x / parts, cta = blockIdx.x / parts;
    long long g = groups <= ctas * kReWarps ? (long long)warp * ctas + cta : cta * kReWarps + warp;
    uint32_t next = marks(g);
    for (; g < groups; g += stride) {
        const uint32_t u = next;
        next = marks(g + stride);
        if (!__any_sync(kFull, u != 0)) continue;
        done += __popc(u);
        bits[lane] = 0;
        int tie_at = 0, ties = 0;   // this lane's pending tie (16 bits of column, the row above), and how many in all
        auto settle = [&] {
            if (lane < ties) {
                const int l = tie_at >> 16, col = tie_at & 0xffff;
                const float *x = A.X + (size_t)(g * rows + l) * d, *r = Rt + (size_t)col * ldr;
                double sum = 0.0;
#pragma unroll 4
                for (int c = 0; c < d; ++c) sum += (double)__ldg(x + c) * (double)__ldg(r + c);
                if (sum >= 0.0) atomicOr(&bits[l * W + (col >> 5)], 1u << (col & 31));
                zeros += sum == 0.0;
            }
            ties = 0;
            __syncwarp();
        };
        for (int l = 0; l < rows; ++l) {
            uint32_t m = wrow == l ? u : 0u;   // row l's marks not yet listed
            if (!__any_sync(kFull, m != 0)) continue;
            const long long row = g * rows + l;
            const float *__restrict__ x = A.X + (size_t)row * d;
            ulonglong2 u0, u1;
            bool zero_row = false;
            if (REG) {
                u0 = x_pairs<VEC, true>(x, 4 * lane, d);
                u1 = x_pairs<VEC, true>(x, 128 + 4 * lane, d);
                zero_row = !__any_sync(kFull, ((u0.x | u0.y | u1.x | u1.y) & kAbs) != 0);
            }
            if (REG && zero_row) {   // against a column of finite values: zero, and not summed (a third of 1e5 x 256: 3.55 ms, 0.29 so)
                uint32_t zero = 0;
                for (uint32_t b = m; b; b &= b - 1)
                    if (__ldg(rn + (lane % W) * 32 + __ffs(b) - 1) < INFINITY) zero |= b & (0u - b);
                zeros += __popc(zero);
                if (zero) atomicOr(&bits[l * W + lane % W], zero);
                m &= ~zero;
                if (!__any_sync(kFull, m != 0)) continue;
            }
            const float xb = 1.25f * roundings * 5.9604644775390625e-8f * __ldg(A.xnorm + row);
            do {
                int hi = 0;
                for (unsigned b; hi <= kReList - 32 && (b = __ballot_sync(kFull, m != 0)) != 0;) {   // one of each word
                    if (m) list[hi + __popc(b & ((1u << lane) - 1u))] = (uint16_t)((lane % W) * 32 + __ffs(m) - 1);
                    m &= m - 1;
                    hi += __popc(b);
                }
                __syncwarp();
                if (lane < 8) list[hi + lane] = list[hi - 1];
                __syncwarp();
                for (int lo = 0; lo < hi; lo += 8) {
                    const uint4 e8 = *reinterpret_cast<const uint4 *>(list + lo);
                    const unsigned e2[4] = {e8.x, e8.y, e8.z, e8.w};
                    const int my_col = list[lo + (lane >> 2)];
                    const float my_rn = __ldg(rn + my_col);
                    float t[8] = {};
                    unsigned long long any = 0;
    #pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (h && lo + 4 >= hi) break;   // (t[4..7] are not looked at)
                        unsigned off[4];
    #pragma unroll
                        for (int i = 0; i < 4; ++i) off[i] = (i & 1 ? e2[2 * h + i / 2] >> 16 : e2[2 * h + i / 2] & 0xffffu) * ldr4;
                        unsigned long long acc[4];
    #pragma unroll
                        for (int i = 0; i < 4; ++i) acc[i] = 0ull;
                        if (REG) {
                            ulonglong2 a[4], b[4];
    #pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                a[i] = __ldg(reinterpret_cast<const ulonglong2 *>(r0 + off[i]));
                                b[i] = __ldg(reinterpret_cast<const ulonglong2 *>(r1 + off[i]));
                            }
    #pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                acc[i] = f2_fma(u0.x, a[i].x, acc[i]);
                                acc[i] = f2_fma(u0.y, a[i].y, acc[i]);
                                acc[i] = f2_fma(u1.x, b[i].x, acc[i]);
                                acc[i] = f2_fma(u1.y, b[i].y, acc[i]);
                            }
                        } else {
    #pragma unroll 2
                            for (int c = 4 * lane; c < ldr; c += 128) {
                                const ulonglong2 xv = x_pairs<VEC, false>(x, c, d);
                                any |= xv.x | xv.y;
                                const char *rc = reinterpret_cast<const char *>(Rt + c);
    #pragma unroll
                                for (int i = 0; i < 4; ++i) {
                                    const ulonglong2 a = __ldg(reinterpret_cast<const ulonglong2 *>(rc + off[i]));
                                    acc[i] = f2_fma(xv.x, a.x, acc[i]);
                                    acc[i] = f2_fma(xv.y, a.y, acc[i]);
                                }
                            }
                        }
    #pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            float e, f;
                            f2_unpack(acc[i], e, f);
                            t[4 * h + i] = e + f;
                        }
                    }
                    if (!REG) zero_row = !__any_sync(kFull, (any & kAbs) != 0);
                    // lane l is left with sum l / 4
    #pragma unroll
                    for (int o = 16, k = 4; o >= 4; o >>= 1, k >>= 1) {
                        const bool high = lane & o;
    #pragma unroll
                        for (int i = 0; i < k; ++i)
                            t[i] = (high ? t[i + k] : t[i]) + __shfl_xor_sync(kFull, high ? t[i] : t[i + k], o);
                    }
                    float s = t[0];
                    s += __shfl_xor_sync(kFull, s, 2);
                    s += __shfl_xor_sync(kFull, s, 1);
                    const bool lead = (lane & 3) == 0 && lo + (lane >> 2) < hi;
                    bool bit = s >= 0.0f;
                    // (a zero row's sum over a finite column is zero: every product is)
                    const unsigned open = __ballot_sync(kFull, lead && !(fabsf(s) > xb * my_rn + tiny));
                    if (open) {
                        if (zero_row && s == 0.0f) zeros += lead;
                        unsigned o = __ballot_sync(kFull, (open >> lane & 1u) && !(zero_row && s == 0.0f));
                        for (const bool ties_likely = __popc(o) > 2; o; o &= o - 1) {
                            const int from = __ffs(o) - 1, c = __shfl_sync(kFull, my_col, from);
                            bool zero = false;
                            const int sg = ties_likely ? 0
                                                       : sign_by_magnitude<VEC>(x, Rt + (size_t)c * ldr, d, ldr,
                                                                                __shfl_sync(kFull, s, from), roundings, &zero);
                            if (lane == from) {
                                bit = sg > 0;
                                zeros += zero;
                            }
                            if (sg == 0) {
                                if (lane == ties) tie_at = l << 16 | c;
                                if (++ties == 32) settle();
                            }
                        }
                    }
                    if (lead && bit) atomicOr(&bits[l * W + (my_col >> 5)], 1u << (my_col & 31));
                }
                __syncwarp();   // the list has been read
            } while (__any_sync(kFull, m != 0));
        }
        if (ties) settle();
        const uint32_t w = bits[lane];
        if (w) A.sig[(size_t)(g * rows + wrow) * words + wword] |= w;
        __syncwarp();
    }
    unsigned long long zs = zeros;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        done += __shfl_xor_sync(kFull, done, o);
        zs += __shfl_xor_sync(kFull, zs, o);
    }
    if (lane == 0 && done) atomicAdd(&A.scratch->counters[2], done);
    if (lane == 0 && zs) atomicAdd(&A.scratch->counters[3], zs);
}

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

struct DenseLayout {
    size_t xh, xl, rh, rl, rt, xn, rn, und, total;
};

DenseLayout dense_layout(long long N, int d0, int bits) {
    const int d = (d0 + BK - 1) / BK * BK;   // K padded to whole stages
    const long long Npad = (N + BM - 1) / BM * BM;
    DenseLayout L;
    size_t o = 0;
    L.xh = o; o = up256(o + (size_t)Npad * d * 2);
    L.xl = o; o = up256(o + (size_t)Npad * d * 2);
    L.rh = o; o = up256(o + (size_t)bits * d * 2);
    L.rl = o; o = up256(o + (size_t)bits * d * 2);
    L.rt = o; o = up256(o + (size_t)bits * d * 4);
    L.xn = o; o = up256(o + (size_t)Npad * 4);
    L.rn = o; o = up256(o + (size_t)bits * 4);
    L.und = o; o = up256(o + (size_t)N * (bits / 8));
    L.total = o;
    return L;
}

bool tc_shape(long long N, int d, int bits) {
    return N > 0 && bits % BN == 0 && d <= 4096 && (N + BM - 1) / BM <= 65535;
}

}  // namespace

extern "C" int blsh_srp_dense_workspace(int64_t N, int32_t d, int32_t bits, size_t *bytes) {
    if (!bytes || N < 0 || d <= 0 || bits <= 0) return BLSH_EINVAL;
    *bytes = tc_shape(N, d, bits) ? dense_layout(N, d, bits).total : 0;
    return BLSH_OK;
}

extern "C" int blsh_srp_dense(blsh_ctx *ctx, const float *X, int64_t N, int32_t d, const float *R, int32_t bits,
                              float margin, uint32_t *sig, void *workspace, size_t workspace_bytes, void *stream) {
    if (!ctx) return BLSH_EINVAL;
    if (!X || !R || !sig) return blsh_fail(ctx, BLSH_EINVAL, "X, R and sig are required");
    if (N < 0 || N >= (1ll << 32) || d <= 0 || bits <= 0 || bits % 32 || bits > 4096 || !(margin == margin))
        return blsh_fail(ctx, BLSH_EINVAL, "bad N, d, bits or margin");
    if (N == 0) return BLSH_OK;
    blsh_device_guard g(ctx->device);
    cudaStream_t s = blsh_stream(stream);
    if (!workspace || !tc_shape(N, d, bits) || !blsh_aligned(X, 16) || !blsh_aligned(R, 16))
        return blsh_srp_dense_simt(ctx, X, N, d, R, bits, sig, s);
    const DenseLayout L = dense_layout(N, d, bits);
    if (workspace_bytes < L.total || !blsh_aligned(workspace, 256)) {
        // widths that are no multiple of 64 need no workspace
        if (d % BK) return blsh_srp_dense_simt(ctx, X, N, d, R, bits, sig, s);
        return blsh_fail(ctx, BLSH_ETRUNC, "workspace needs %zu bytes, 256-byte aligned", L.total);
    }
    const int KT = (d + BK - 1) / BK;
    // the margin must cover the tensor-core error: split 3.1 * 2^-16, FP32
    // accumulation of 3 Kpad products at 2^-22 each, with a 25% slack
    const float rigorous = 1.25f * (4.0f * 1.52587890625e-5f + 3.0f * (float)(KT * BK) * 2.384185791015625e-7f);
    const float m = margin > rigorous ? margin : rigorous;
    unsigned char *ws = (unsigned char *)workspace;
    const long long Npad = (N + BM - 1) / BM * BM;
    uint32_t *und = (uint32_t *)(ws + L.und);
    const int r_blocks = bits / kPrepCols;
    const unsigned x_blocks = (unsigned)((Npad + 7) / 8 < 65535ll * 8 ? (Npad + 7) / 8 : 65535ll * 8);
    const bool vec = d % 4 == 0;
    blsh_time_start(ctx, s);
    (vec ? srp_dense_prep<true> : srp_dense_prep<false>)<<<r_blocks + x_blocks, 256, 0, s>>>(
        X, N, Npad, d, KT, ws + L.xh, ws + L.xl, (float *)(ws + L.xn), R, bits, ws + L.rh, ws + L.rl,
        (float *)(ws + L.rn), (float *)(ws + L.rt), r_blocks);
    BLSH_LAUNCHED(ctx, "srp_dense_prep");
    const size_t smem = (size_t)STAGES * STAGE_BYTES + 1024 + (size_t)bits * sizeof(float);
    const size_t smem_max = (size_t)STAGES * STAGE_BYTES + 1024 + 4096 * sizeof(float);   // bits <= 4096
    static std::atomic<unsigned long long> opted{0};
    if (ctx->device < 64 && !((opted.load() >> ctx->device) & 1ull)) {
        BLSH_CUDA(ctx, cudaFuncSetAttribute(srp_dense_tc_persistent, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)smem_max));
        opted.fetch_or(1ull << ctx->device);
    }
    const long long tiles = (long long)(bits / BN) * (Npad / BM);
    const unsigned grid = (unsigned)(tiles < ctx->sm_count ? tiles : ctx->sm_count);
    blsh_time_start(ctx, s);
    srp_dense_tc_persistent<<<grid, kTcThreads, smem, s>>>(ws + L.xh, ws + L.xl, ws + L.rh, ws + L.rl,
                                                          (float *)(ws + L.xn), (float *)(ws + L.rn), N, d, bits, m,
                                                          sig, und, tiles, ctx->scratch);
    BLSH_LAUNCHED(ctx, "srp_dense_tc_persistent");
    blsh_time_start(ctx, s);
    const int part_words = bits % 1024 == 0 ? 32 : bits % 512 == 0 ? 16 : 8, parts = bits / (32 * part_words);
    const RecheckArgs A = {und, X, (const float *)(ws + L.rt), (const float *)(ws + L.xn), (const float *)(ws + L.rn), N,
                           d, KT * BK, bits, part_words, sig, ctx->scratch};
    const long long groups = (N * part_words + 31) / 32;
    const long long copies = ctx->sm_count / parts > 0 ? ctx->sm_count / parts : 1;   // CTAs a part
    const unsigned re_grid = (unsigned)((groups < copies ? groups : copies) * parts);
    if (d <= 256)
        (vec ? srp_dense_recheck_kernel<true, true> : srp_dense_recheck_kernel<false, true>)<<<re_grid, 32 * kReWarps, 0,
                                                                                             s>>>(A);
    else
        (vec ? srp_dense_recheck_kernel<true, false> : srp_dense_recheck_kernel<false, false>)<<<
            re_grid, 32 * kReWarps, 0, s>>>(A);
    BLSH_LAUNCHED(ctx, "srp_dense_recheck_kernel");
    return BLSH_OK;
}
