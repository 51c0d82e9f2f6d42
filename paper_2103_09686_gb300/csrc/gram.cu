// Three-point descriptor (sm_103a): the quadratic reduction of the ensemble, Eq. s3,
//     S_bar3(r_a, r_b) = (1/N) sum_x e_x(r_a) e_x(r_b),   e_x(r) = f((M_x + M_{x+r}) / 2),
// i.e. the Gram matrix E^T E / N of the N x K ensemble (paper, Sec. 3.2.2-3.2.4 and the
// footnote of Sec. 3.4), and the gradient of a loss on it.
//
//   ens_kernel      e and f' never leave the chip except as the GEMM operands: E (N x K)
//                   and E^T (K x N), each split into two FP16 parts, e s = hi + lo with
//                   hi = fp16(e s), lo = fp16(e s - hi) (22 significant bits; s = 1 for the
//                   soft threshold, whose f is bounded, and a power of two bringing max |M|
//                   into [1/2, 1) for f(x) = x);
//   tc_gemm_kernel  C = A B^T on the 5th-generation tensor cores: tcgen05.mma kind::f16
//                   from shared memory, FP32 accumulators in TMEM drained every 256-512
//                   reduction steps into FP32 registers, three products
//                   hi*hi + hi*lo + lo*hi per k-step (the dropped lo*lo is below 2^-22 of the
//                   product), operands staged by TMA (128-byte swizzled K-major layout), one
//                   thread issues the MMAs and commits them to an mbarrier per stage; the
//                   epilogue undoes the operands' scales exactly;
//                   S_bar3 = Et Et^T w/N (upper-triangle 128 x 128 tiles, mirrored);
//   tc_gemm_pair_kernel  the same for W^T = (2/N) G E^T as E G^T with a transposed epilogue:
//                   256 x 256 tiles, each on a pair of SMs (cta_group::2);
//   g3_split_kernel G = w * gscale * (D3 - D3_des) symmetrised (or the upstream gradient),
//                   scaled by the power of two that brings max |G| (g3_absmax_kernel) into
//                   [1/2, 1), split like E;
//   s3_gather_kernel g_y = sum_r 1/2 [W(r, y) f'(a_y(r)) + W(r, y - r) f'(a_{y-r}(r))]
//                   (weight 1 at r = 0), the two ends of every shift vector.
// Every wait on an mbarrier is bounded; a timeout sets an error flag that the host reads.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cstdio>
#include <mutex>

#include "common.cuh"

namespace dmcr {

// C = scale * A B^T on the tensor cores (see tc_gemm_kernel): operands as TMA tensor maps
struct GemmArgs {
    CUtensorMap ta_hi, ta_lo, tb_hi, tb_lo;
    int M, N, K;
    float scale;
    const float* amaxA;     // operand scale sources (null: unscaled); C *= 2^(eA + eB)
    const float* amaxB;
    float* C;
    int64_t ldc;
    int Mvalid, Nvalid;
    const int* done;
    int* err;
};

// the same with plain device pointers (host side)
struct GemmOperands {
    const uint16_t *Ah, *Al, *Bh, *Bl;   // FP16 bit patterns
    int64_t lda, ldb;
    int M, N, K;
    float scale;
    const float* amaxA;
    const float* amaxB;
    float* C;
    int64_t ldc;
    int mode;               // 1 symmetric Gram (upper tiles, mirrored), 2 C[n][m]
    int Mvalid, Nvalid;
    const int* done;
    int* err;
};

namespace {

// A CTA holds 128 rows of a tile; GK reduction steps per stage, three stages.  Both kernels stage
// 128 rows of A and of B, hi and lo, 64 KB.
constexpr int GM = 128, GK = 64;
constexpr int OP_TILE = GM * GK * 2;                   // one FP16 operand tile (128 rows of 128 bytes), 16 KB
constexpr int STAGE_BYTES = 4 * OP_TILE;               // A hi, A lo, B hi, B lo
constexpr int GSTAGES = 3;
constexpr size_t GEMM_SMEM = (size_t)GSTAGES * STAGE_BYTES + 1024 + 256;
constexpr uint32_t BUF_COLS = 256, TMEM_COLS = 512;    // two accumulator buffers
constexpr int EC = 128;                                // accumulator columns of one epilogue thread
// Gram: 4 epilogue warps; a buffer holds hi*hi and, 128 columns further, the small cross terms
// hi*lo + lo*hi.  Pair: 8 epilogue warps; a buffer holds all three products of 256 columns and
// is drained twice as often.
constexpr int GRAM_EPI = 4, GRAM_FLUSH = 8;
constexpr int PAIR_EPI = 8, PAIR_FLUSH = 4;
// instruction descriptor, kind::f16: D F32 (bits 4-5 = 1), A and B F16 (bits 7-9, 10-12 = 0),
// both K-major (bits 15, 16 = 0), N >> 3 at bits 17-22, M >> 4 at bits 24-28
__host__ __device__ constexpr uint32_t idesc_f16(int m, int n) { return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24); }
// The tensor core adds into its FP32 accumulator without round-to-nearest: over a long
// reduction the error is biased toward zero (~4e-8 relative per accumulation measured on
// GB300).  So TMEM accumulates at most FLUSH k-blocks before the partial sums are added,
// rounded to nearest, into FP32 registers.
constexpr uint32_t WAIT_LIMIT = 1u << 22;
constexpr unsigned long long WAIT_NS = 4000000000ull;


__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// 2-D tiled TMA load of one box into shared memory, completion counted on an mbarrier
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
        "[%4];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// bounded wait (tries, and WAIT_NS of time) for the completion of the mbarrier phase with the
// given parity; CLUSTER: the other CTA of the pair arrives on it
template <bool CLUSTER = false>
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
    const uint32_t addr = smem_u32(bar);
    unsigned long long start = 0;
    for (uint32_t i = 0; i < WAIT_LIMIT; ++i) {
        uint32_t ok;
        if constexpr (CLUSTER)
            asm volatile(
                "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                "selp.b32 %0, 1, 0, p;\n\t}"
                : "=r"(ok)
                : "r"(addr), "r"(parity)
                : "memory");
        else
            asm volatile(
                "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                "selp.b32 %0, 1, 0, p;\n\t}"
                : "=r"(ok)
                : "r"(addr), "r"(parity)
                : "memory");
        if (ok) return true;
        if (i % 1024 == 1023) {
            unsigned long long now;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
            if (start == 0) start = now;
            else if (now - start > WAIT_NS) return false;
        }
    }
    return false;
}
// arrive on the barrier at the same place in the pair's first CTA
__device__ __forceinline__ void mbar_arrive_first(uint64_t* bar) {
    asm volatile(
        "{\n\t.reg .b32 ra;\n\tmapa.shared::cluster.u32 ra, %0, 0;\n\t"
        "mbarrier.arrive.release.cluster.shared::cluster.b64 _, [ra];\n\t}" ::"r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// whole warp: allocate all TMEM columns, address written to shared memory; PAIR: one warp of each
// CTA of the pair
template <bool PAIR>
__device__ __forceinline__ void tmem_alloc(uint32_t* slot) {
    if constexpr (PAIR) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
}
template <bool PAIR>
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr) {
    if constexpr (PAIR)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(TMEM_COLS) : "memory");
    else
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(TMEM_COLS) : "memory");
}

// shared-memory matrix descriptor, K-major with the 128-byte swizzle: each operand row is
// one 128-byte line (64 FP16) whose 16-byte chunks are stored at chunk ^ (row % 8); atoms of
// 8 rows (1024 bytes, 1024-byte aligned) follow each other at SBO = 1024; LBO is unused by
// this layout (encoded 1); descriptor version 1, layout type 2 (SWIZZLE_128B).  A k-step of
// 16 FP16 starts 32 bytes further into the line.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) |
           (2ull << 61);
}

template <bool PAIR>
__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    if constexpr (PAIR)
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
            "l"(a), "l"(b), "r"(idesc), "r"(acc)
            : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
            "l"(a), "l"(b), "r"(idesc), "r"(acc)
            : "memory");
}

// arrive on the barrier (PAIR: at the same place in both CTAs) when every earlier MMA of this
// thread has completed
template <bool PAIR>
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    if constexpr (PAIR)
        asm volatile(
            "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
                smem_u32(bar)),
            "h"((uint16_t)3)
            : "memory");
    else
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                         smem_u32(bar))
                     : "memory");
}

// 32 lanes x 16 columns of 32 bits: thread i of the warp gets lane (lane base + i)
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

// x = hi + lo to 22 significant bits (both FP16, round to nearest)
__device__ __forceinline__ void split_f16(float x, uint16_t& hi, uint16_t& lo) {
    const __half h = __float2half_rn(x);
    hi = __half_as_ushort(h);
    lo = __half_as_ushort(__float2half_rn(x - __half2float(h)));
}

// exponent e of the scale 2^-e that maps max |x| = *amax into [1/2, 1); 0 without a source,
// for 0 and for non-finite maxima
__device__ __forceinline__ int scale_exp(const float* amax) {
    if (amax == nullptr) return 0;
    const float a = *amax;
    if (!(a > 0.f) || !isfinite(a)) return 0;
    int e;
    frexpf(a, &e);
    return e;
}

}  // namespace

// ------------------------------------------------------------------------- GEMM

// C = scale 2^(eA + eB) A B^T with A (M x K) and B (N x K) row-major (K contiguous), each given
// as FP16 hi + lo through four TMA tensor maps (boxes 64 x 128, 128-byte swizzle; rows past the
// end read as zero).  K a multiple of 64.
//
// Warp roles of both kernels: warp EPI (one lane) loads the stages with TMA; warp EPI + 1 (one
// lane) issues the MMAs and commits them; warps 0 .. EPI - 1 drain the TMEM accumulators every
// FLUSH k-blocks into FP32 registers (warp w reads TMEM lanes 32 (w % 4) .. + 31 and columns
// 128 (w / 4) .. + 127; TMEM is double-buffered) and write the tile.  Barriers: full[s] (TMA
// bytes landed), empty[s] (MMAs done reading stage s), tfull[b] (period finished in TMEM buffer
// b), tempty[b] (buffer b read), mdone (every MMA finished).

// all k-blocks of one tile into the stages; kb0 counts the k-blocks of the CTA's earlier tiles
__device__ __forceinline__ bool load_tile(const GemmArgs& g, uint8_t* gsm, uint64_t* full, uint64_t* empty, int nk,
                                          int row_a, int row_b, int64_t kb0, int64_t& issued) {
    for (int kb = 0; kb < nk; ++kb) {
        const int64_t q = kb0 + kb;
        const int s = (int)(q % GSTAGES);
        if (q >= GSTAGES && !mbar_wait(&empty[s], (uint32_t)((q / GSTAGES) - 1) & 1)) return false;
        uint8_t* st = gsm + s * STAGE_BYTES;
        mbar_expect_tx(&full[s], STAGE_BYTES);
        const int k0 = kb * GK;
        tma_load_2d(st, &g.ta_hi, k0, row_a, &full[s]);
        tma_load_2d(st + OP_TILE, &g.ta_lo, k0, row_a, &full[s]);
        tma_load_2d(st + 2 * OP_TILE, &g.tb_hi, k0, row_b, &full[s]);
        tma_load_2d(st + 3 * OP_TILE, &g.tb_lo, k0, row_b, &full[s]);
        issued = q + 1;
    }
    return true;
}

// No copy of a CTA may still be in flight when it exits, after a give-up as well: wait (bounded)
// for the bytes of the stages it actually started.  Each stage's barrier has begun no phase after
// the one waited on here, so the parity is unambiguous.
__device__ __forceinline__ bool drain_loads(uint64_t* full, int64_t issued) {
    bool ok = true;
    for (int64_t q = issued > GSTAGES ? issued - GSTAGES : 0; q < issued; ++q)
        if (!mbar_wait(&full[q % GSTAGES], (uint32_t)(q / GSTAGES) & 1)) ok = false;
    return ok;
}

// The Gram: A = B, M = N, only tiles bn >= bm of 128 x 128, written to C[m][n] and C[n][m] where
// m, n < Mvalid.  One tile a CTA: the upper triangle holds few (136 at 1985 shifts).  Bound by
// what an SM reads from L2 and shared memory (64 KB a stage for 768 cycles of MMA), so hi*hi and
// hi*lo are one MMA of 256 columns over the adjacent hi and lo tiles of B: A is read twice per
// k-step, not three times.  The tile goes through shared memory on its way to the rows of C, so
// both halves of the matrix are written in lines.  2048 x 2048 over 16384 / 4096 positions: 143 / 45
// us (75 / 63 % of the tensor pipe; three MMAs of 128 columns and rows written by lane: 170 / 62).
__global__ void __launch_bounds__(32 * (GRAM_EPI + 2), 1) tc_gemm_kernel(const __grid_constant__ GemmArgs g) {
    extern __shared__ __align__(1024) uint8_t gsm_raw[];
    // the swizzle atoms need 1024-byte aligned tiles
    uint8_t* gsm = gsm_raw + ((1024 - (smem_u32(gsm_raw) & 1023)) & 1023);
    uint64_t* full = reinterpret_cast<uint64_t*>(gsm + GSTAGES * STAGE_BYTES);
    uint64_t* empty = full + GSTAGES;
    uint64_t* tfull = empty + GSTAGES;
    uint64_t* tempty = tfull + 2;
    uint64_t* mdone = tempty + 2;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(mdone + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int s = 0; s < GSTAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], GRAM_EPI * 32);
        }
        mbar_init(mdone, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == GRAM_EPI + 1) tmem_alloc<false>(tslot);
    // the upper triangle row by row: (bm, bn >= bm)
    const int tiles = g.N / GM;
    int bm = 0, t = (int)blockIdx.x;
    while (t >= tiles - bm) {
        t -= tiles - bm;
        ++bm;
    }
    const int bn = bm + t;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;
    dep_wait();
    dep_trigger();
    const bool skip = g.done != nullptr && *g.done;
    const int nk = skip ? 0 : g.K / GK;
    const int nper = (nk + GRAM_FLUSH - 1) / GRAM_FLUSH;
    bool ok = true;

    if (warp == GRAM_EPI) {
        if (lane == 0) {
            int64_t issued = 0;
            ok = load_tile(g, gsm, full, empty, nk, bm * GM, bn * GM, 0, issued);
            if (!drain_loads(full, issued)) ok = false;
        }
        __syncwarp();
    } else if (warp == GRAM_EPI + 1) {
        // ---- MMA issuer
        if (lane == 0) {
            for (int kb = 0; kb < nk; ++kb) {
                const int s = kb % GSTAGES;
                const int p = kb / GRAM_FLUSH, buf = p & 1;
                // TMEM buffer buf was last used by period p - 2: wait until it was read
                if (kb % GRAM_FLUSH == 0 && p >= 2) ok = mbar_wait(&tempty[buf], ((p / 2) - 1) & 1);
                if (ok) ok = mbar_wait(&full[s], (kb / GSTAGES) & 1);
                if (!ok) break;
                tc_fence_after();
                const uint32_t st = smem_u32(gsm + s * STAGE_BYTES);
                const uint32_t t_acc = tmem + (uint32_t)buf * BUF_COLS;
#pragma unroll
                for (int ks = 0; ks < GK / 16; ++ks) {
                    const uint32_t off = ks * 32;   // 16 FP16 = 32 bytes per k-step
                    const uint64_t ah = smem_desc_sw128(st + off), al = smem_desc_sw128(st + OP_TILE + off);
                    const uint64_t b = smem_desc_sw128(st + 2 * OP_TILE + off);   // hi, then lo: 256 rows
                    mma_f16<false>(t_acc, ah, b, idesc_f16(GM, 256), (kb % GRAM_FLUSH != 0) || ks != 0);
                    mma_f16<false>(t_acc + GM, al, b, idesc_f16(GM, GM), 1);
                }
                mma_commit<false>(&empty[s]);
                if (kb % GRAM_FLUSH == GRAM_FLUSH - 1 || kb == nk - 1) mma_commit<false>(&tfull[buf]);
            }
            // TMEM is freed below: first every MMA issued above (all of them, also after a
            // give-up of this thread or of another role) must have finished writing it.  A
            // commit tracks every earlier tcgen05 operation of this thread.
            mma_commit<false>(mdone);
            if (!mbar_wait(mdone, 0)) ok = false;
        }
        __syncwarp();
    } else {
        // ---- epilogue
        float acc[EC];
#pragma unroll
        for (int c = 0; c < EC; ++c) acc[c] = 0.f;
        for (int p = 0; p < nper; ++p) {
            const int buf = p & 1;
            // warp-uniform decision: tcgen05.ld below is .sync.aligned
            ok = __all_sync(0xffffffffu, mbar_wait(&tfull[buf], (p / 2) & 1));
            if (!ok) break;
            tc_fence_after();
            const uint32_t t_acc = tmem + (uint32_t)buf * BUF_COLS + ((uint32_t)(32 * warp) << 16);
#pragma unroll
            for (int c = 0; c < EC; c += 16) {
                float v[16], w[16];
                tmem_ld16(t_acc + (uint32_t)c, v);
                tmem_ld16(t_acc + GM + (uint32_t)c, w);
#pragma unroll
                for (int j = 0; j < 16; ++j) acc[c + j] += v[j] + w[j];
            }
            tc_fence_before();
            mbar_arrive(&tempty[buf]);
        }
        if (!skip) {
            const int r = 32 * warp + lane, m = bm * GM + r;
            // undo the operands' power-of-two scales together with the output scale (exact)
            const float scale = ldexpf(g.scale, scale_exp(g.amaxA) + scale_exp(g.amaxB));
            // the last period's barrier: every stage has been read, its memory is free (given up
            // on: this warp's part of it is not used)
            float* tile = reinterpret_cast<float*>(gsm);
            if (ok) {
#pragma unroll
                for (int c = 0; c < EC; ++c) {
                    const int n = bn * GM + c;
                    const float x = scale * acc[c];
                    tile[r * (GM + 1) + c] = x;
                    if (bm != bn && m < g.Mvalid && n < g.Nvalid) g.C[(int64_t)n * g.ldc + m] = x;
                }
                __syncwarp();
                for (int q = 0; q < 32; ++q) {
                    const int mr = 32 * warp + q;
                    if (bm * GM + mr >= g.Mvalid) break;
                    float* C = g.C + (int64_t)(bm * GM + mr) * g.ldc + bn * GM;
#pragma unroll
                    for (int c = lane; c < GM; c += 32)
                        if (bn * GM + c < g.Nvalid) C[c] = tile[mr * (GM + 1) + c];
                }
            }
        }
    }
    if (!ok && g.err != nullptr) atomicExch(g.err, 1);
    // the MMA issuer reaches this barrier only after its last commit arrived (or its bounded
    // wait for it ran out), and the epilogue warps after their last TMEM read
    tc_fence_before();
    __syncthreads();
    if (warp == GRAM_EPI + 1) tmem_dealloc<false>(tmem);
}

// C[n][m] = scale A B^T where m < Mvalid and n < Nvalid; N a multiple of 256.  A pair of CTAs
// (one cluster, two SMs) owns a 256 x 256 tile: each holds 128 rows of A, half of B's rows and
// the accumulators of its 128 rows, and the first CTA's MMAs (cta_group::2) work on both.  Per
// SM a stage of 64 KB feeds 1536 cycles of MMA (one CTA alone on 128 x 256 needs 96 KB for them,
// what L2 can deliver to an SM at best).  The kernel is persistent: the pairs walk the tiles (B
// tiles fastest: the pairs in flight share a few row blocks of A and sweep the whole of B, which
// stays in L2), and while the epilogue warps write a tile the next one's stages and first
// periods are under way.  16384 / 4096 x 2048 over 2048: 231 / 72 us (80 / 74 % of the tensor
// pipe; one CTA on a 128 x 256 tile, one tile a CTA: 306 / 100).
// The copies signal each CTA's own barriers; the second CTA's MMA warp passes its full[s] on to
// the first CTA's pfull[s].  Commits arrive in both CTAs; tempty[b] of the first CTA counts the
// epilogue warps of both.
__global__ void __launch_bounds__(32 * (PAIR_EPI + 2), 1) tc_gemm_pair_kernel(const __grid_constant__ GemmArgs g) {
    extern __shared__ __align__(1024) uint8_t gsm_raw[];
    uint8_t* gsm = gsm_raw + ((1024 - (smem_u32(gsm_raw) & 1023)) & 1023);
    uint64_t* full = reinterpret_cast<uint64_t*>(gsm + GSTAGES * STAGE_BYTES);
    uint64_t* empty = full + GSTAGES;
    uint64_t* pfull = empty + GSTAGES;
    uint64_t* tfull = pfull + GSTAGES;
    uint64_t* tempty = tfull + 2;
    uint64_t* mdone = tempty + 2;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(mdone + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = (int)cluster_rank();
    if (tid == 0) {
        for (int s = 0; s < GSTAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
            mbar_init(&pfull[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], 2 * PAIR_EPI);
        }
        mbar_init(mdone, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == PAIR_EPI + 1) tmem_alloc<true>(tslot);
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    tc_fence_after();
    const uint32_t tmem = *tslot;
    dep_wait();
    dep_trigger();
    const bool skip = g.done != nullptr && *g.done;
    const int nk = g.K / GK;
    const int nper = (nk + PAIR_FLUSH - 1) / PAIR_FLUSH;
    const int tilesN = g.N / 256;
    const int tiles = skip ? 0 : (g.M + 255) / 256 * tilesN;
    const int first = (int)(blockIdx.x / 2), pairs = (int)(gridDim.x / 2);
    bool ok = true;

    if (warp == PAIR_EPI) {
        // ---- TMA producer
        if (lane == 0) {
            int64_t issued = 0, kb0 = 0;
            for (int t = first; ok && t < tiles; t += pairs, kb0 += nk)
                ok = load_tile(g, gsm, full, empty, nk, t / tilesN * 256 + rank * GM, t % tilesN * 256 + rank * GM, kb0,
                               issued);
            if (!drain_loads(full, issued)) ok = false;
            // the commits that arrive here from the first CTA have to land before the exit, too
            for (int64_t q = issued > GSTAGES ? issued - GSTAGES : 0; q < issued; ++q)
                if (!mbar_wait(&empty[q % GSTAGES], (uint32_t)(q / GSTAGES) & 1)) ok = false;
        }
        __syncwarp();
    } else if (warp == PAIR_EPI + 1) {
        if (lane == 0 && rank == 0) {
            // ---- MMA issuer
            int64_t q = 0, p = 0;      // k-blocks and periods so far
            for (int t = first; ok && t < tiles; t += pairs) {
                for (int kb = 0; kb < nk; ++kb, ++q) {
                    const int s = (int)(q % GSTAGES), buf = (int)(p & 1);
                    const uint32_t par = (uint32_t)(q / GSTAGES) & 1;
                    // TMEM buffer buf was last used by period p - 2: wait until both CTAs read it
                    if (kb % PAIR_FLUSH == 0 && p >= 2) ok = mbar_wait<true>(&tempty[buf], (uint32_t)((p / 2) - 1) & 1);
                    if (ok) ok = mbar_wait(&full[s], par);
                    if (ok) ok = mbar_wait<true>(&pfull[s], par);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t st = smem_u32(gsm + s * STAGE_BYTES);
                    const uint32_t t_acc = tmem + (uint32_t)buf * BUF_COLS;
#pragma unroll
                    for (int ks = 0; ks < GK / 16; ++ks) {
                        const uint32_t off = ks * 32;   // 16 FP16 = 32 bytes per k-step
                        const uint64_t ah = smem_desc_sw128(st + off), al = smem_desc_sw128(st + OP_TILE + off);
                        const uint64_t bh = smem_desc_sw128(st + 2 * OP_TILE + off);
                        const uint64_t bl = smem_desc_sw128(st + 3 * OP_TILE + off);
                        mma_f16<true>(t_acc, ah, bh, idesc_f16(256, 256), (kb % PAIR_FLUSH != 0) || ks != 0);
                        mma_f16<true>(t_acc, ah, bl, idesc_f16(256, 256), 1);
                        mma_f16<true>(t_acc, al, bh, idesc_f16(256, 256), 1);
                    }
                    mma_commit<true>(&empty[s]);
                    if (kb % PAIR_FLUSH == PAIR_FLUSH - 1 || kb == nk - 1) {
                        mma_commit<true>(&tfull[buf]);
                        ++p;
                    }
                }
            }
            // as in the Gram: every MMA issued above must have finished before the exit
            mma_commit<true>(mdone);
            if (!mbar_wait(mdone, 0)) ok = false;
        } else if (lane == 0) {
            // ---- the second CTA's stages are announced to the first
            int64_t q = 0;
            for (int t = first; ok && t < tiles; t += pairs)
                for (int kb = 0; kb < nk; ++kb, ++q) {
                    const int s = (int)(q % GSTAGES);
                    ok = mbar_wait(&full[s], (uint32_t)(q / GSTAGES) & 1);
                    if (!ok) break;
                    mbar_arrive_first(&pfull[s]);
                }
            if (!mbar_wait(mdone, 0)) ok = false;
        }
        __syncwarp();
    } else {
        // ---- epilogue
        const int quad = warp & 3, half = warp >> 2;
        // undo the operands' power-of-two scales together with the output scale (exact)
        const float scale = ldexpf(g.scale, scale_exp(g.amaxA) + scale_exp(g.amaxB));
        int64_t p = 0;
        for (int t = first; ok && t < tiles; t += pairs) {
            float acc[EC];
#pragma unroll
            for (int c = 0; c < EC; ++c) acc[c] = 0.f;
            for (int i = 0; i < nper; ++i, ++p) {
                const int buf = (int)(p & 1);
                ok = __all_sync(0xffffffffu, mbar_wait(&tfull[buf], (uint32_t)(p / 2) & 1));
                if (!ok) break;
                tc_fence_after();
                const uint32_t t_acc =
                    tmem + (uint32_t)buf * BUF_COLS + (uint32_t)(EC * half) + ((uint32_t)(32 * quad) << 16);
#pragma unroll
                for (int c = 0; c < EC; c += 16) {
                    float v[16];
                    tmem_ld16(t_acc + (uint32_t)c, v);
#pragma unroll
                    for (int j = 0; j < 16; ++j) acc[c + j] += v[j];
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_first(&tempty[buf]);
            }
            const int m = t / tilesN * 256 + rank * GM + 32 * quad + lane;
            const int n0 = t % tilesN * 256 + EC * half;
            if (ok && m < g.Mvalid) {
                float* C = g.C + (int64_t)n0 * g.ldc + m;
#pragma unroll
                for (int c = 0; c < EC; ++c, C += g.ldc)
                    if (n0 + c < g.Nvalid) *C = scale * acc[c];
            }
        }
    }
    if (!ok && g.err != nullptr) atomicExch(g.err, 1);
    // neither CTA frees its TMEM, or exits, before both are through
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    tc_fence_after();
    if (warp == PAIR_EPI + 1) tmem_dealloc<true>(tmem);
    cluster_sync();
}

// ------------------------------------------------------------------------- ensemble

// shift k of the canonical half window -> (rz, ry, rx); inverse of canon_index (32-bit: the
// half window holds at most 2^14 shifts here)
__device__ __forceinline__ void decode_shift(const LevelGeom& g, int k, int& rz, int& ry, int& rx) {
    const int Px = g.P[2], Py = g.P[1];
    const int wx = 2 * Px + 1, wy = 2 * Py + 1;
    if (k <= Px) {
        rz = 0; ry = 0; rx = k;
        return;
    }
    k -= Px + 1;
    if (k < Py * wx) {
        rz = 0; ry = 1 + k / wx; rx = k % wx - Px;
        return;
    }
    k -= Py * wx;
    rz = 1 + k / (wy * wx);
    k %= wy * wx;
    ry = k / wx - Py;
    rx = k % wx - Px;
}

// position coordinates of a level (z, y, c), 32-bit (levels hold < 2^31 positions)
struct Pos3 {
    int z, y, c;
};

__device__ __forceinline__ Pos3 pos_of(const LevelGeom& g, int64_t x) {
    const int n12 = (int)(g.n[1] * g.n[2]), n2 = (int)g.n[2];
    const int xi = (int)x;
    Pos3 p;
    p.z = xi / n12;
    const int r = xi - p.z * n12;
    p.y = r / n2;
    p.c = r - p.y * n2;
    return p;
}

// v + d wrapped into [0, n) for |d| <= n (windows never exceed half a level)
__device__ __forceinline__ int wrap_add(int v, int d, int n) {
    int w = v + d;
    w = w >= n ? w - n : w;
    return w < 0 ? w + n : w;
}

// s = sigma(alpha (a - 0.75)) for a = (u + v) / 2, exact form (any finite range)
__device__ __forceinline__ float sig_pair(const ThreshConst& tc, float u, float v) {
    float e;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(fmaf(-tc.kappa, u + v, tc.cexp)));
    float s;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(e + 1.0f));
    return s;
}

// One block: 128 positions x 64 shifts; a lane owns four consecutive positions and a warp eight
// consecutive shifts, whose partners it reaches by stepping along rx (the row is found again only
// where (rz, ry) changes).  E^T rows (shift-major) are written as 8 bytes per lane, 256 per warp;
// E rows (position-major) go through shared memory, 16-byte chunks of eight shifts stored at
// chunk ^ (position / 4 % 8) (conflict-free both ways), and are written as 128-byte lines.
// Padding entries are 0.  Bound by the instruction rate and, close to it, by the stores
// (8 bytes an entry): 16384 x 1985: 52 us
// (5.2 TB/s; 64 x 32 blocks with an index computed per entry: 116 us).
constexpr int ENS_X = 128, ENS_K = 64;

// the pair (a, b) split into FP16 hi and lo words (a in the lower half)
__device__ __forceinline__ void split_pair(float a, float b, uint32_t& hi, uint32_t& lo) {
    const __half2 h = __floats2half2_rn(a, b);
    const float2 f = __half22float2(h);
    const __half2 l = __floats2half2_rn(a - f.x, b - f.y);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
}

template <bool IDENTITY>
__global__ void __launch_bounds__(256, 3) ens_kernel(const __grid_constant__ S3Job j, const __grid_constant__ ThreshConst tc) {
    dep_wait();
    dep_trigger();
    if (j.done != nullptr && *j.done) return;
    __shared__ uint4 th[ENS_X * 8], tl[ENS_X * 8];
    const LevelGeom& g = j.g;
    if (blockIdx.x == 0 && threadIdx.x == 0) j.amax[0] = 0.f;     // max |G| starts here
    // f(x) = x: e is bounded by max |M|, scaled into [-1, 1); the soft f is bounded by ~1.03
    const float sE = IDENTITY ? ldexpf(1.f, -scale_exp(j.amax + 1)) : 1.f;
    const unsigned xb = (unsigned)(j.Npad / ENS_X);
    const int64_t x0 = (int64_t)(blockIdx.x % xb) * ENS_X, k0 = (int64_t)(blockIdx.x / xb) * ENS_K;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n0 = (int)g.n[0], n1 = (int)g.n[1], n2 = (int)g.n[2];
    const int64_t xa = x0 + 4 * lane;
    const int64_t ka = k0 + 8 * warp;
    const float* __restrict__ field = j.field;
    bool in[4];
    float u[4];
    Pos3 p[4];
    int row[4], col[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        in[q] = xa + q < g.N;
        p[q] = pos_of(g, in[q] ? xa + q : 0);
        u[q] = in[q] ? field[xa + q] : 0.f;
    }
    int rz = 0, ry = 0, rx = 0;
    if (ka < j.K) decode_shift(g, (int)ka, rz, ry, rx);
    auto start_row = [&]() {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            row[q] = (wrap_add(p[q].z, rz, n0) * n1 + wrap_add(p[q].y, ry, n1)) * n2;
            col[q] = wrap_add(p[q].c, rx, n2);
        }
    };
    start_row();
    uint32_t hw[4][4], lw[4][4];        // [position][pair of shifts]
    uint32_t ph[2], pl[2];              // the pair's first shift, positions in pairs
    uint2* Eth = reinterpret_cast<uint2*>(j.Eth + ka * j.Npad + xa);
    uint2* Etl = reinterpret_cast<uint2*>(j.Etl + ka * j.Npad + xa);
    const int64_t step = j.Npad / 4;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        float e[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            e[q] = 0.f;
            if (ka + i < j.K) {
                const float v = field[row[q] + col[q]];
                e[q] = IDENTITY ? 0.5f * (u[q] + v) * sE : fmaf(tc.c1, sig_pair(tc, u[q], v), tc.c3);
                if (!in[q]) e[q] = 0.f;
            }
            const unsigned c = (unsigned)col[q] + 1u;
            col[q] = (int)min(c, c - (unsigned)n2);
        }
        if (++rx > g.P[2]) {
            rx = -g.P[2];
            if (++ry > g.P[1]) {
                ry = -g.P[1];
                ++rz;
            }
            if (ka + i + 1 < j.K) start_row();
        }
        uint32_t h[2], l[2];
        split_pair(e[0], e[1], h[0], l[0]);
        split_pair(e[2], e[3], h[1], l[1]);
        Eth[i * step] = make_uint2(h[0], h[1]);
        Etl[i * step] = make_uint2(l[0], l[1]);
        if (i % 2 == 0) {
            ph[0] = h[0], ph[1] = h[1], pl[0] = l[0], pl[1] = l[1];
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const unsigned sel = q % 2 ? 0x7632u : 0x5410u;
                hw[q][i / 2] = __byte_perm(ph[q / 2], h[q / 2], sel);
                lw[q][i / 2] = __byte_perm(pl[q / 2], l[q / 2], sel);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int o = (4 * lane + q) * 8 + (warp ^ (lane & 7));
        th[o] = make_uint4(hw[q][0], hw[q][1], hw[q][2], hw[q][3]);
        tl[o] = make_uint4(lw[q][0], lw[q][1], lw[q][2], lw[q][3]);
    }
    __syncthreads();
    // E rows: 128 positions x 8 chunks
    const int c = threadIdx.x & 7;
    for (int pp = threadIdx.x >> 3; pp < ENS_X; pp += 32) {
        const int64_t o = (x0 + pp) * j.Kpad + k0 + 8 * c;
        const int t = pp * 8 + (c ^ ((pp >> 2) & 7));
        *reinterpret_cast<uint4*>(j.Eh + o) = th[t];
        *reinterpret_cast<uint4*>(j.El + o) = tl[t];
    }
}

// G(a, b) = w * gscale * sym(D3 - D3_des) on the level's K x K block; d<G, E^T E>/dE =
// E (G + G^T), so G is symmetrised (the loss gradient already is symmetric).  A block holds
// a 32 x 32 tile; the transposed entries come through shared memory, so both reads are
// coalesced, and v is symmetric: a block covers the tiles (ta, tb) and (tb, ta), ta <= tb, from
// one read of both.  Returns v(a0 + i, b0 + tx) for i = ty, ty + 8, ... in v[4] (0 outside K x K).
__device__ __forceinline__ float g3_delta(const S3Job& j, int64_t a, int64_t b) {
    return j.src[a * j.K + b] - (j.sub != nullptr ? j.sub[a * j.K + b] : 0.f);
}

__device__ __forceinline__ void g3_tile(const S3Job& j, int64_t a0, int64_t b0, float (*tt)[33], float (&v)[4]) {
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    float d[4], m[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int64_t i = ty + 8 * q;
        d[q] = (a0 + i < j.K && b0 + tx < j.K) ? g3_delta(j, a0 + i, b0 + tx) : 0.f;
        m[q] = (b0 + i < j.K && a0 + tx < j.K) ? g3_delta(j, b0 + i, a0 + tx) : 0.f;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) tt[tx][ty + 8 * q] = m[q];
    __syncthreads();
    const float sc = j.weight * (j.sc != nullptr ? j.sc->gscale : 1.f);
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = sc * 0.5f * (d[q] + tt[ty + 8 * q][tx]);
}

// block -> tile pair (ta <= tb) of the upper triangle, columns in order: tb (tb + 1) / 2 + ta
__device__ __forceinline__ void g3_pair(int64_t t, int64_t& ta, int64_t& tb) {
    tb = (int64_t)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
    while (tb * (tb + 1) / 2 > t) --tb;
    while ((tb + 1) * (tb + 2) / 2 <= t) ++tb;
    ta = t - tb * (tb + 1) / 2;
}

// max |v| of a block's values into *out (non-negative floats order like their bit patterns;
// *out starts at 0)
__device__ __forceinline__ void block_absmax(float m, float* out) {
    __shared__ float sh[8];
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, sh[w]);
        atomicMax(reinterpret_cast<int*>(out), __float_as_int(m));
    }
}

// one pair of 32 x 32 tiles of G per block (K = 1985: 12 us; each tile on its own 18)
__global__ void __launch_bounds__(256) g3_absmax_kernel(const __grid_constant__ S3Job j) {
    dep_wait();
    dep_trigger();
    if (j.done != nullptr && *j.done) return;
    __shared__ float tt[32][33];
    int64_t ta, tb;
    g3_pair(blockIdx.x, ta, tb);
    float v[4];
    g3_tile(j, ta * 32, tb * 32, tt, v);
    float m = 0.f;
    for (int q = 0; q < 4; ++q) m = fmaxf(m, fabsf(v[q]));
    block_absmax(m, j.amax);
}

// f(x) = x: max |M| of the level's field, the bound of |e|
__global__ void __launch_bounds__(256) field_absmax_kernel(const __grid_constant__ S3Job j) {
    dep_wait();
    dep_trigger();
    if (j.done != nullptr && *j.done) return;
    float m = 0.f;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < j.g.N; i += (int64_t)gridDim.x * blockDim.x)
        m = fmaxf(m, fabsf(j.field[i]));
    block_absmax(m, j.amax + 1);
}

// G scaled by 2^-eG (max |G| into [1/2, 1)) and split into FP16 hi + lo, one pair of 32 x 32
// tiles of Kpad x Kpad per block (zero padding; K = 1985: 14 us, each tile on its own 20)
__global__ void __launch_bounds__(256) g3_split_kernel(const __grid_constant__ S3Job j) {
    dep_wait();
    dep_trigger();
    if (j.done != nullptr && *j.done) return;
    __shared__ float tt[32][33];
    int64_t ta, tb;
    g3_pair(blockIdx.x, ta, tb);
    float v[4];
    g3_tile(j, ta * 32, tb * 32, tt, v);
    const int eG = scale_exp(j.amax);
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    // the second tile is the transpose of the first
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) tt[tx][ty + 8 * q] = v[q];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int r = ty + 8 * q;
        uint16_t hi, lo;
        split_f16(ldexpf(v[q], -eG), hi, lo);
        const int64_t i = (ta * 32 + r) * j.Kpad + tb * 32 + tx;
        j.Gh[i] = hi;
        j.Gl[i] = lo;
        split_f16(ldexpf(tt[r][tx], -eG), hi, lo);
        const int64_t t = (tb * 32 + r) * j.Kpad + ta * 32 + tx;
        j.Gh[t] = hi;
        j.Gl[t] = lo;
    }
}

// g_y = sum_k c_k [W(k, y) f'(a_y(r_k)) + W(k, y - r_k) f'(a_{y - r_k}(r_k))], c_0 = 1/2 (the two
// terms coincide at r = 0), c_k = 1/2 otherwise; f' = c1 alpha s (1 - s), or 1 for f(x) = x.
// Block (position block, shift chunk of S3_SHIFTS): per-chunk partials, summed in a fixed order
// by the gradient assembly.  The chunk's shifts come in canonical order (rx fastest, then ry,
// then rz): the partner columns are stepped along rx, the rows rebuilt where (rz, ry) changes;
// four shifts per step, their loads issued together.  Bound by the instruction rate (four
// special-function operations a term): 16384 x 1985 61 us, 127 with 64-bit indexes.
template <bool IDENTITY>
__global__ void __launch_bounds__(256, 5) s3_gather_kernel(const __grid_constant__ S3Job j, const __grid_constant__ ThreshConst tc) {
    dep_wait();
    dep_trigger();
    if (j.done != nullptr && *j.done) return;
    const LevelGeom& g = j.g;
    const int y = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (y >= g.N) return;
    const int kA = (int)blockIdx.y * S3_SHIFTS;
    const int nk = (int)min((int64_t)S3_SHIFTS, j.K - kA);
    const float* __restrict__ field = j.field;
    const float* __restrict__ W = j.W + (int64_t)kA * j.Npad;
    const int n0 = (int)g.n[0], n1 = (int)g.n[1], n2 = (int)g.n[2];
    const float my = field[y];
    const Pos3 py = pos_of(g, y);
    int rz, ry, rx, rowp, rowm, cp, cm;
    decode_shift(g, kA, rz, ry, rx);
    auto rows = [&]() {
        rowp = (wrap_add(py.z, rz, n0) * n1 + wrap_add(py.y, ry, n1)) * n2;
        rowm = (wrap_add(py.z, -rz, n0) * n1 + wrap_add(py.y, -ry, n1)) * n2;
        cp = wrap_add(py.c, rx, n2);
        cm = wrap_add(py.c, -rx, n2);
    };
    rows();
    auto next = [&]() {
        if (++rx > g.P[2]) {
            rx = -g.P[2];
            if (++ry > g.P[1]) {
                ry = -g.P[1];
                ++rz;
            }
            rows();
        } else {
            const unsigned c = (unsigned)cp + 1u;
            cp = (int)min(c, c - (unsigned)n2);
            cm = cm == 0 ? n2 - 1 : cm - 1;
        }
    };
    // W f' without the constant factor c1 alpha
    auto term = [&](float w, float u, float v) {
        if (IDENTITY) return w;
        const float s = sig_pair(tc, u, v);
        return w * fmaf(-s, s, s);
    };
    float acc = 0.f;
    constexpr int U = 4;
    int k = 0;
    for (; k + U <= nk; k += U, W += U * j.Npad) {
        float vp[U], vm[U], w1[U], w2[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int ym = rowm + cm;                           // y - r
            vp[u] = IDENTITY ? 0.f : field[rowp + cp];          // y + r
            vm[u] = IDENTITY ? 0.f : field[ym];
            w1[u] = W[u * j.Npad + y];
            w2[u] = W[u * j.Npad + ym];
            next();
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            acc += term(w1[u], my, vp[u]);
            acc += term(w2[u], vm[u], my);
        }
    }
    for (; k < nk; ++k, W += j.Npad) {
        const int ym = rowm + cm;
        acc += term(W[y], my, field[rowp + cp]);
        acc += term(W[ym], field[ym], my);
        next();
    }
    j.part[(int64_t)blockIdx.y * g.N + y] = IDENTITY ? 0.5f * acc : 0.5f * tc.c1 * tc.alpha * acc;
}

// ------------------------------------------------------------------------- launchers

void set_gram_attributes() {
    cudaFuncSetAttribute(tc_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GEMM_SMEM);
    cudaFuncSetAttribute(tc_gemm_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GEMM_SMEM);
}

__global__ void set_flag_kernel(int* flag, int v) {
    dep_wait();
    dep_trigger();
    if (flag != nullptr) *flag = v;
}

// cuTensorMapEncodeTiled through the runtime's driver entry point (no libcuda link)
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// rows x cols FP16 row-major (row stride ld elements), boxes of box_rows rows x 64 columns
bool make_map(CUtensorMap* m, const uint16_t* base, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (enc == nullptr) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * sizeof(uint16_t)};
    const cuuint32_t box[2] = {(cuuint32_t)GK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<uint16_t*>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool gram_ready() { return tensor_map_encoder() != nullptr; }

// Pairs of CTAs that are resident at once (one CTA an SM; an SM without a partner stays out): the
// persistent kernel's grid, since a pair that had to wait would run its tiles after all others.
int resident_pairs(cudaLaunchConfig_t cfg) {
    static std::mutex mu;
    static int known[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1;
    std::lock_guard<std::mutex> lk(mu);
    if (known[dev] == 0) {
        int n = 0;
        cfg.gridDim = dim3(2);
        if (cudaOccupancyMaxActiveClusters(&n, tc_gemm_pair_kernel, &cfg) != cudaSuccess || n < 1) {
            cudaGetLastError();
            n = 32;
        }
        known[dev] = n;
    }
    return known[dev];
}

// mode 1: the Gram (A = B, M = N multiples of 128); mode 2: C[n][m] on pairs of SMs
void launch_tc_gemm(const GemmOperands& o, cudaStream_t s) {
    const int64_t tm = o.M / GM;
    if (tm <= 0 || o.N <= 0) return;
    GemmArgs a{};
    const bool ok = make_map(&a.ta_hi, o.Ah, o.M, o.K, o.lda, GM) && make_map(&a.ta_lo, o.Al, o.M, o.K, o.lda, GM) &&
                    make_map(&a.tb_hi, o.Bh, o.N, o.K, o.ldb, GM) && make_map(&a.tb_lo, o.Bl, o.N, o.K, o.ldb, GM);
    if (!ok) {
        // no valid tensor map: never launch TMA on it; report through the error word
        launch_dep(set_flag_kernel, 1, 1, 0, s, o.err, 2);
        return;
    }
    a.M = o.M; a.N = o.N; a.K = o.K;
    a.scale = o.scale;
    a.amaxA = o.amaxA;
    a.amaxB = o.amaxB;
    a.C = o.C;
    a.ldc = o.ldc;
    a.Mvalid = o.Mvalid; a.Nvalid = o.Nvalid;
    a.done = o.done;
    a.err = o.err;
    if (o.mode == 1) {
        launch_dep(tc_gemm_kernel, (unsigned)(tm * (tm + 1) / 2), 32 * (GRAM_EPI + 2), GEMM_SMEM, s, a);
        return;
    }
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.blockDim = dim3(32 * (PAIR_EPI + 2));
    cfg.dynamicSmemBytes = GEMM_SMEM;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const int64_t tiles = (tm + 1) / 2 * (o.N / 256);
    const int64_t pairs = std::min<int64_t>(tiles, resident_pairs(cfg));
    cfg.gridDim = dim3((unsigned)(2 * pairs));
    cfg.numAttrs = 2;
    cudaLaunchKernelEx(&cfg, tc_gemm_pair_kernel, a);
}

constexpr int ABSMAX_BLOCKS = 512;

// E and E^T of one level (f(x) = x: after the bound of |e|)
void launch_ensemble(const S3Job& j, const ThreshConst& tc, cudaStream_t s) {
    const unsigned blocks = (unsigned)((j.Npad / ENS_X) * (j.Kpad / ENS_K));
    if (tc.identity) {
        launch_dep(set_flag_kernel, 1, 1, 0, s, reinterpret_cast<int*>(j.amax + 1), 0);
        const int64_t fb = std::min<int64_t>(ABSMAX_BLOCKS, (j.g.N + 255) / 256);
        launch_dep(field_absmax_kernel, (unsigned)fb, 256, 0, s, j);
        launch_dep(ens_kernel<true>, blocks, 256, 0, s, j, tc);
    } else {
        launch_dep(ens_kernel<false>, blocks, 256, 0, s, j, tc);
    }
}

void launch_s3_forward(const S3Job& j, const ThreshConst& tc, int* err, cudaStream_t s) {
    launch_ensemble(j, tc, s);
    GemmOperands a{};
    a.Ah = j.Eth; a.Al = j.Etl; a.Bh = j.Eth; a.Bl = j.Etl;
    a.amaxA = a.amaxB = tc.identity ? j.amax + 1 : nullptr;
    a.lda = a.ldb = j.Npad;
    a.M = a.N = (int)j.Kpad;
    a.K = (int)j.Npad;
    a.scale = (float)((double)j.weight / (double)j.g.N);
    a.C = j.desc;
    a.ldc = j.K;
    a.mode = 1;
    a.Mvalid = a.Nvalid = (int)j.K;
    a.done = j.done;
    a.err = err;
    launch_tc_gemm(a, s);
}

void launch_s3_backward(const S3Job& j, const ThreshConst& tc, int* err, cudaStream_t s) {
    if (j.ens) launch_ensemble(j, tc, s);
    const int64_t tk = (j.K + 31) / 32, tp = j.Kpad / 32;
    launch_dep(g3_absmax_kernel, (unsigned)(tk * (tk + 1) / 2), 256, 0, s, j);
    launch_dep(g3_split_kernel, (unsigned)(tp * (tp + 1) / 2), 256, 0, s, j);
    GemmOperands a{};
    a.Ah = j.Eh; a.Al = j.El; a.Bh = j.Gh; a.Bl = j.Gl;
    a.amaxA = tc.identity ? j.amax + 1 : nullptr;
    a.amaxB = j.amax;
    a.lda = j.Kpad;
    a.ldb = j.Kpad;
    a.M = (int)j.Npad;
    a.N = (int)j.Kpad;
    a.K = (int)j.Kpad;
    a.scale = (float)(2.0 / (double)j.g.N);
    a.C = j.W;
    a.ldc = j.Npad;
    a.mode = 2;
    a.Mvalid = (int)j.Npad;
    a.Nvalid = (int)j.Kpad;
    a.done = j.done;
    a.err = err;
    launch_tc_gemm(a, s);
    const dim3 grid((unsigned)((j.g.N + 255) / 256), (unsigned)((j.K + S3_SHIFTS - 1) / S3_SHIFTS));
    if (tc.identity) launch_dep(s3_gather_kernel<true>, grid, 256, 0, s, j, tc);
    else launch_dep(s3_gather_kernel<false>, grid, 256, 0, s, j, tc);
}

}  // namespace dmcr
