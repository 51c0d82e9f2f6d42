// Shared declarations of the dmcr CUDA library (kernels + C ABI).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <memory>
#include <vector>

#include "scalars.h"
#include "sep_basis.h"

namespace dmcr {

constexpr int T = 8;            // shifts per thread (forward) / positions per strip (adjoint)
constexpr int TX = 32;          // tile width in positions (fastest axis)
constexpr int FWD_THREADS = 128;
constexpr int ADJ_THREADS = 128;   // 32 row pairs (lane, lane + 32) x 4 strips of 8 positions
constexpr int ADJ_ROWS = 64;       // adjoint tile rows
constexpr int GBLOCK = 48;         // coefficient floats per block of 8 shifts (packed pairs)
constexpr int S3_SHIFTS = 32;      // three-point gradient gather: shifts per partial sum

// offset of C_m inside a coefficient block: (C_m, C_m, C_m+1, C_m+1) after the 8 (A, A, B, B)
__host__ __device__ inline int gblock_c(int m) { return 4 * T + 2 * m; }
constexpr int NPEN_BLOCKS = 512;   // most blocks of the loss statistics of one instance

// Double-float sums: an FP32 pair hi + lo carries about 48 significant bits.  FP64
// arithmetic is slow on this part, and the reductions below sit on the critical path of
// every iteration, so they add double-floats in fixed orders instead.
struct DF {
    float hi, lo;
};

// a + b exactly as hi + lo (Knuth's two-sum; no ordering of |a|, |b| needed); commutative
__device__ __forceinline__ DF df_two_sum(float a, float b) {
    const float s = a + b;
    const float bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}

__device__ __forceinline__ DF df_add(DF a, DF b) {
    const DF s = df_two_sum(a.hi, b.hi);
    const float lo = s.lo + (a.lo + b.lo);
    const float hi = s.hi + lo;
    return {hi, lo - (hi - s.hi)};
}

// fixed-order sums over the block (blockDim.x a multiple of 32): xor butterflies in each warp, then
// over the warp results in warp 0, all NV values side by side; the results are valid in warp 0.
// sh holds NV entries for every warp.
template <int NV>
__device__ __forceinline__ void block_sums_df(DF (&v)[NV], DF* sh) {
    auto warp_sums = [&]() {
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int i = 0; i < NV; ++i)
                v[i] = df_add(v[i], DF{__shfl_xor_sync(0xffffffffu, v[i].hi, o), __shfl_xor_sync(0xffffffffu, v[i].lo, o)});
    };
    warp_sums();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    __syncthreads();   // sh may still be read by a previous call
    if (lane == 0)
#pragma unroll
        for (int i = 0; i < NV; ++i) sh[warp * NV + i] = v[i];
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) v[i] = lane < nw ? sh[lane * NV + i] : DF{0.f, 0.f};
        warp_sums();
    }
}
__device__ __forceinline__ DF block_sum_df(DF v, DF* sh) {
    DF a[1] = {v};
    block_sums_df(a, sh);
    return a[0];
}

// Programmatic dependent launch.  A kernel launched with launch_dep may start while its
// predecessor in the stream still runs; dep_wait() returns once every earlier kernel has
// completed and its writes are visible, and dep_trigger() lets the successor start.  Every
// kernel triggers only after its own wait, so what a kernel reads before dep_wait() may be
// anything written at least two launches earlier (the segment tables), and nothing else.
__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dep_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
inline void launch_dep(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

constexpr int MAX_DYN_SMEM = 200 * 1024;   // dynamic shared memory limit of the correlation kernels
constexpr int SMS = 152;           // what the splits of work that depend on the free part of the chip aim at
constexpr int MAX_PHASES = 8;      // phase fields of one problem (their ordered pairs each get a block)

// One multigrid level, every field handled as 3-D (2-D fields have n[0] = 1, P[0] = 0).
struct LevelGeom {
    int64_t n[3];
    int64_t N;
    int P[3];
    int NB;           // rx blocks of T covering [-P2, P2]
    int64_t NG;       // shift groups (rz, ry, b) of the half window
    int64_t Khalf;
    int64_t NGT;      // NG * T (columns of one forward partial row)
    // forward tiling
    int TY;           // tile rows
    int PPB;          // planes per block
    int tilesY, tilesX, planeChunks;
    int64_t fwdTiles; // planeChunks * tilesY * tilesX
    int fwdGroupBlocks;
    // adjoint tiling
    int adjTilesY, adjTilesX;
    int64_t adjTiles;  // n[0] * adjTilesY * adjTilesX
    int nZc, nYc, RZ, RY;   // shift chunks over rz and ry
    int RYS;                // ry rows staged in shared memory at a time (RY may be larger: rounds)
    int nXc, NBc;           // shift chunks over the rx blocks: NBc blocks of T per chunk
    int nChunks;
    int fft;          // 1: this level runs on the FFT path (identity threshold / binary target)
};

// Soft-threshold constants in the product form used on the device:
//   P = E'_x E_y,  E_y = 2^(-kappa M_y),  E'_x = 2^(cexp - kappa M_x)
//   s = 1/(1+P) = sigma(alpha (a - 0.75)),  f = c1 s + c3.
struct ThreshConst {
    float kappa;     // (alpha/2) log2(e)
    float cexp;      // 0.75 alpha log2(e)
    float c1, c3;
    float alpha;
    float lim;       // product form when |kappa M| <= lim everywhere in a block
    float beta;      // c3 / c1: f = c1 (s + beta)
    int identity;    // f(x) = x
};

struct LossParams {
    int mode;           // 0 norm, 1 squared
    float lambda0;
    int bc_on;
    int64_t Ktot;
    int64_t N;          // finest pixel count
    float tol_rel;      // <=0: no stopping test
    int check_every;
    float lr, beta1, beta2;
    int max_iters;
    int recon;          // 1: update iteration / Adam bookkeeping
};

struct FinalArgs {
    const int* tier;             // separable levels (sep.cu): below SEP_TIERS, sparts replaces parts
    const float* sparts[8];      // their gradient, one field per level
    int ndim;
    int levels;
    int64_t n1[3];               // finest sizes (3-D embedded)
    const float* parts[8];       // adjoint partials per level
    int nChunks[8];
    int64_t Nl[8];
    int64_t nl[8][3];
    const float* field;          // finest field (penalty), may be null when no penalty
    const Scalars* sc;           // pen_coef (null: no penalty)
    float* grad_out;             // may be null
    float* M;                    // Adam: field to update (null: no Adam)
    float* m;
    float* v;
    float beta1, beta2, eps;
};

// ---------------------------------------------------------------- segment tables
// A fused launch covers several (instance, level) segments; every segment owns the
// contiguous block range [blockStart, next blockStart) of a 1-D grid and the kernels find
// their segment by binary search.  Tables live in device memory (written by blob_kernel).
struct LossSeg {
    LossParams lp;
    const float4* sums;         // block sums of (D - D_des)^2 and D_des^2 (hi, lo each)
    const float4* excess;       // block sums of the squared box excess (hi, lo)
    int nsum, nexc;
    Scalars* sc;
    float* loss_out;
    float* history;
};
struct FwdSeg {
    LevelGeom g;
    const float* field;     // tails of the pairs (x)
    const float* tip;       // tips of the pairs (x + r): the same field, or another phase's
    float* partial;
    const int* gate;        // gated launches only: run when *gate >= SEP_TIERS
    unsigned* next;         // gated launches only: the first block that nobody has taken (prep_kernel sets it to 0)
    const int* done;
    int64_t blockStart;
};
struct RedSeg {
    LevelGeom g;
    const float* partial;
    float* desc;
    const int* gate;        // gated launches only: run when *gate >= SEP_TIERS
    unsigned* next;         // gated launches only: the first block that nobody has taken (prep_kernel sets it to 0)
    const int* done;
    float scale;             // w_l / N_l
    // loss: this segment's target, its block sums (one per block), the instance's loss and the
    // number of blocks that leave sums for it; null: no loss, or statistics by stats_kernel
    const float* target;
    float4* sums;
    const LossSeg* loss;
    int arrive;
    // box excess of the field in `nexc` extra blocks of this segment (0: elsewhere or none)
    int nexc;
    float4* excess;
    const float* field;
    int64_t fieldN, excChunk;
    int64_t blockStart;
};
// Gradient coefficients of one level and phase pair: G(r) from the residuals or the upstream
// gradient (see coef_value in corr.cu).
struct CoefSrc {
    const float* src;       // dL/dS (or S - S_des) of the block (a, b), shifts r of the half window
    const float* sub;
    const float* src2;      // the block (b, a), which holds -r; src2 = src, sub2 = sub for a = b
    const float* sub2;
    const Scalars* sc;
    float scale;
    const float* tsum;      // corrected descriptor: sum_{k >= 1} (src - sub) of the block, else null
    float q;                // corrected descriptor: 2 f(1/2)^2
};
struct AdjSeg {
    LevelGeom g;
    const float* field;     // own positions y (the gradient's field)
    const float* tip;       // partners y + r: the same field, or another phase's
    CoefSrc c;
    float* part;
    const int* gate;        // gated launches only: run when *gate >= SEP_TIERS
    unsigned* next;         // gated launches only: the first block that nobody has taken (prep_kernel sets it to 0)
    const int* done;
    int64_t blockStart;
};
// dense coefficient grid of an FFT level
struct GSeg {
    LevelGeom g;
    CoefSrc c;
    float* Gd;
    const int* done;
    int64_t blockStart;
};
// Corrected two-point descriptor (App. A, Eq. s2rfroms2rbar), one (instance, level) block:
// forward, the block is mapped in place, S_tilde(k) = (S_bar(k) - q S_bar(0)) / (1 - q) for
// k >= 1; backward, tsum = sum_{k >= 1} (src - sub) feeds the transposed map in gcoef.
struct TildeSeg {
    float* desc;
    const float* src;
    const float* sub;
    float* tsum;
    int64_t K;
    float q;
    const int* done;
    int64_t blockStart;
};
struct RestrictSeg {
    int ndim;
    int64_t c[3];               // coarse sizes (3-D embedded)
    const float* fine;
    float* coarse;
    const int* done;
    int64_t blockStart;
};
// Pyramid of one instance (one block range over all its phases): every coarser level that a
// tile of the finest grid determines, and with `tiers` the range tier of each block's values.
constexpr int PREP_TILE2 = 32, PREP_TILE3 = 16;      // tile edge: 2-D 32 x 32, 3-D 16 x 16 x 16
constexpr int PREP_LEVELS2 = 5, PREP_LEVELS3 = 4;    // coarser levels of one tile
constexpr int PREP_BLOCKS = 256;                     // blocks per instance at most
struct PrepSeg {
    int ndim, coarse;            // coarser levels to build here
    int phases, nblk;
    int n[3];                    // finest sizes (3-D embedded)
    const float* field;
    float* lv[PREP_LEVELS2];     // level 2, 3, ... (phases stacked)
    int* tiers;                  // separable path: one word per block, null otherwise: its tier, and from bit 8
                                 // on one bit per phase that shows a value of at least SEP_WEAK
    float* sums;                 // separable path: sum of the block's values, [block][phase]
    unsigned* next;              // separable path: the gated segments' counters, set to 0 (nnext of them)
    int nnext;
    int ntier;
    float lo[8], hi[8];          // its ranges
    float4* excess;              // box excess: sum of squares per block (hi, lo), null: not wanted
    const int* done;
    int64_t blockStart;
};
struct PenSeg {
    const float* field;      // null: no box penalty
    int64_t N;
    const float* desc;
    const float* target;
    int64_t K;
    float4 *sums, *excess;   // nblk each
    const LossSeg* loss;
    const int* done;
    int nblk;                // blocks of this instance: a function of its own sizes only
};
struct FinalSeg {
    FinalArgs a;
    const int* done;
    int64_t blockStart;
};
// Three-point descriptor, one (instance, level) (gram.cu).  K = half-window shifts, Kpad =
// K rounded up to 256, Npad = the level's position count rounded up to 128.
struct S3Job {
    LevelGeom g;
    const float* field;     // this level's field
    int64_t K, Kpad, Npad;
    // GEMM operands as FP16 bit patterns: x s = hi + lo (hi = fp16(x s), lo = fp16(x s - hi)),
    // s a power of two that brings max |x| into [1/2, 1) (E: f(x) = x only; G: always)
    uint16_t *Eh, *El;      // E (Npad x Kpad)
    uint16_t *Eth, *Etl;    // E^T (Kpad x Npad)
    float* W;               // W^T (Kpad x Npad)
    uint16_t *Gh, *Gl;      // G (Kpad x Kpad)
    float* amax;            // [0] max |G|, [1] max |field| (f(x) = x): the scales' sources
    float* desc;            // this level's K x K block of the descriptor (w * S_bar3)
    const float* src;       // G = weight * (sc ? gscale : 1) * (src - sub): src = desc (loss) or
    const float* sub;       //   the upstream gradient (VJP, sub = null, sc = null)
    const Scalars* sc;
    float weight;
    float* part;            // this level's gradient
    const int* done;
    int ens;                // backward: build E first (no forward ran in this call)
    int* err;               // set on a tensor-core wait timeout
};

// FFT path, one (instance, level) (fft.cu).
struct FftAxis {
    int n, nrad;
    unsigned char rad[16];
    double2* tw;              // tw[t] = exp(-2 pi i t / n)
};
struct FftArgs {
    int n0, n1, n2, nh;       // sizes; nh = n2 / 2 + 1 columns of the half spectrum
    int P0, P1, P2, NB;
    int64_t N;
    FftAxis ax[3];
    int Lx, Ly, Ll;           // lines per block: rows (row pairs), middle axis, last axis
    int Lv, Lw;               // the window's rows and middle axis
    const float* field;
    double2 *X, *U, *V;       // half spectrum of the field; window planes (3-D) and rows
    double* sq;               // sum M^2 of the row blocks
    int nsq;
    double* dc;               // sum_r A(r)
    const float* Gd;          // dense coefficient grid (plane 0 is A)
    float weight;
    int mode;                 // 0 identity threshold, 1 soft threshold of a binary field
    double fh2;               // f(1/2)^2
    float* desc;
    float* part;
    int x_ready;              // X holds the whole transform (the descriptor ran in this call)
};

// ---------------------------------------------------------------- separable path (sep.cu)
constexpr int SEP_THREADS = 512;    // threads of the transform kernels
constexpr int SEP_BLOCK_PTS = 8 * SEP_THREADS;   // points a block holds in registers (power-of-two axes)
constexpr int SEP_ROW_THREADS = 256;   // threads of the feature and gradient kernels
constexpr int SEP_SLOTS = 8;        // feature pairs a row block holds side by side at most
constexpr int SEP_FAST_PHASES = 3;  // phases whose spectra fit behind the line buffers of sep_mul
constexpr int SEP_MAX_N = 2048;     // longest axis
constexpr int64_t SEP_MAX_POINTS = 1 << 28;   // points of one grid (32-bit offsets)
constexpr int SEP_MAX_RAD = 12;
constexpr int SEP_OWN = 8;          // points of a column group one thread owns (at most 4096 per block)
constexpr int SEP_MAX_SMEM = 222 * 1024;

struct SepAxis {
    int n, nrad;
    int fast;                 // log2 n for powers of two 16 .. SEP_MAX_N, else 0
    unsigned short rad[SEP_MAX_RAD];
};

// line pitch (float2 elements) of a column group of L adjacent columns: padded length, and
// pitch = 16 / L (mod 16), so that the L columns of one position lie in different banks
__host__ __device__ inline int sep_pitch(int n, int L) {
    const int p = n - 1 + ((n - 1) >> 4) + 1;
    const int want = L >= 16 ? 1 : 16 / L;
    return p + ((want - p) % 16 + 16) % 16;
}

// one (instance, level)
struct SepLevel {
    int n0, n1, n2;
    int P0, P1, P2;
    int phases, maxPairs;
    int64_t N, Khalf;
    SepAxis ax[3];
    const float* field;       // this level's field(s)
    float2 *Z, *Q;            // spectra of the features, products: phases x maxPairs grids (one phase: Q = Z)
    float2 *U, *V;            // window spectra (3-D: [r0][y][x]; [row][x]), one per ordered phase pair
    int64_t strideU, strideV;
    float2* dc;               // scaleD sum_k s_k conj(Z^a_k(0)) Z^b_k(0) per phase pair (hi, lo)
    const float* msum;        // PrepSeg.sums: [range block][phase]
    float invN1;              // 1 / points of the finest level
    float* center;            // per phase, the value that the features vanish at (sep_feat)
    float* phi;               // sums of F(M^a, center_b) by the warps of sep_feat, nphi per phase pair; null: not wanted
    int nphi;
    float* gsum;              // sum of G over the window, one per phase pair
    int* tiers;               // tiers of the range blocks (PrepSeg.tiers)
    int ntiers;
    int* tier;                // the instance's tier
    int first;                // finest level: writes *tier
    int keep;                 // one phase, forward and backward in one call: sep_power leaves its spectra in Z
    int rowsF, rowsW, colsY, colsL;
    int parts;                // sums of sep_power (over a share of the pairs each) that sep_desc adds, strideV apart
    float* desc;
    double scaleD;            // w / N^2
    const float* src;         // gradient coefficients: scaleG (gscale) (src - sub)
    const float* sub;
    const Scalars* sc;
    const float* tsum;        // corrected descriptor
    float q, scaleG;
    int fuse;                 // one phase, loss and gradient in one call: sep_desc goes on to the rows of G
    const LossSeg* loss;      // sep_desc leaves the loss' sums (`sums`, one per block of the instance) and
    float4* sums;             //   its last block finishes the loss; null: no loss, or statistics elsewhere
    int sumStart, arrive;     // this level's first block sum of phase pair 0; blocks in all
    float* part;              // this level's gradient, one field per phase
    const int* done;
};

struct SepItem {
    int level, a, b;
    int parts;                // sep_power, sep_mul: blocks that share the pairs of one group of columns
    int64_t blockStart;
    const int* tier;
    const int* done;
};

struct SepTables {
    const SepLevel* level;
    const float2* coef;
    SepTier tier[SEP_TIERS];
    float alpha, c1, c3;      // of the threshold (ThreshConst)
};

enum SepKernel {
    SEP_FEAT, SEP_FFT_Y, SEP_POWER, SEP_POWER_PH, SEP_INV_Y, SEP_DESC, SEP_GX, SEP_GY, SEP_MUL, SEP_MUL_PH, SEP_IFFT_Y,
    SEP_GRAD, SEP_KERNELS
};

const float2* sep_device_coef(const SepBasis& b);
bool sep_axis(int64_t n, SepAxis& ax);
double sep_axis_cost(const SepAxis& ax);
int sep_cols(const SepAxis& ax, bool wide, int phases);
int sep_window_rows(const SepAxis& ax);
int sep_feature_rows(const SepAxis& ax, int64_t rows);
size_t sep_smem_feat(const SepLevel& lv);
size_t sep_smem_window(const SepLevel& lv);
size_t sep_smem_y(const SepLevel& lv);
size_t sep_smem_last(const SepLevel& lv, bool mul);
void launch_sep(SepKernel k, const SepTables& tb, const SepItem* items, int nitem, int64_t blocks, size_t smem,
                cudaStream_t s);
void set_sep_attributes();

// ---------------------------------------------------------------- launchers
void launch_blob(const void* host, size_t bytes, void* dst, cudaStream_t s);
void launch_prep(const PrepSeg* segs, int nseg, int64_t blocks, cudaStream_t s);
void launch_restrict(const RestrictSeg* segs, int nseg, int64_t blocks, cudaStream_t s);
void launch_restrict_one(int ndim, const int64_t nf[3], const float* fine, float* coarse, cudaStream_t s);
void launch_prolongate(int ndim, const int64_t nc[3], const float* coarse, float* fine, int mode,
                       cudaStream_t s);
void launch_corr_fwd(const FwdSeg* segs, int nseg, int64_t blocks, size_t smem, const ThreshConst& tc,
                     cudaStream_t s);
void launch_fwd_reduce(const RedSeg* segs, int nseg, int64_t blocks, cudaStream_t s);
// the same for the segments whose gate says so (fields outside every separable range)
void launch_corr_fwd_gated(const FwdSeg* segs, int nseg, int64_t blocks, size_t smem, const ThreshConst& tc,
                           cudaStream_t s);
void launch_fwd_reduce_gated(const RedSeg* segs, int nseg, int64_t blocks, cudaStream_t s);
void launch_corr_adj_gated(const AdjSeg* segs, int nseg, int64_t blocks, size_t smem, const ThreshConst& tc,
                           cudaStream_t s);
void launch_penalty(const PenSeg* segs, int nseg, int maxblk, cudaStream_t s);
int stats_blocks(int64_t K, int64_t N);
void launch_gcoef(const GSeg* segs, int nseg, int64_t blocks, const ThreshConst& tc, cudaStream_t s);
void launch_tilde_map(const TildeSeg* segs, int nseg, int64_t blocks, cudaStream_t s);
void launch_tilde_sum(const TildeSeg* segs, int nseg, cudaStream_t s);
void launch_corr_adj(const AdjSeg* segs, int nseg, int64_t blocks, size_t smem, const ThreshConst& tc,
                     cudaStream_t s);
// sub = threads per position: 1, or FIN_SUB for segments of fields below FIN_SUB_BELOW positions
void launch_final(const FinalSeg* segs, int nseg, int64_t blocks, int sub, cudaStream_t s);
void launch_init_uniform(float* field, int64_t count, uint64_t seed, cudaStream_t s);
void launch_round_field(const float* src, float* dst, int64_t count, cudaStream_t s);
void set_kernel_attributes();
void set_gram_attributes();
bool gram_ready();   // the TMA tensor-map encoder is available
void launch_s3_forward(const S3Job& j, const ThreshConst& tc, int* err, cudaStream_t s);
void launch_s3_backward(const S3Job& j, const ThreshConst& tc, int* err, cudaStream_t s);
void set_fft_attributes();
void fft_axis(int len, FftAxis& ax);
int fft_lines_per_block(int len, bool strided);
void fft_window_lines(FftArgs& g);
int fft_row_blocks(const FftArgs& g);
void launch_fft_descriptor(const FftArgs& g, cudaStream_t s);
void launch_fft_vjp(const FftArgs& g, cudaStream_t s);
size_t fwd_smem_bytes(const LevelGeom& g);
size_t adj_smem_bytes(const LevelGeom& g);
float gcoef_scale(const LevelGeom& g, const ThreshConst& tc, float weight);

constexpr int RED_K = 32;      // shifts per fwd_reduce block
constexpr int GCOEF_TH = 256;  // entries per gcoef block
constexpr int ELEM_TH = 256;   // pixels per restrict block; threads per final block
constexpr int FIN_SUB = 8;     // gradient assembly of a small field: threads per position (each sums
                               // every 8th chunk)
constexpr int64_t FIN_SUB_BELOW = 1 << 16;   // fields of fewer positions use FIN_SUB threads each
// Positions of one thread of the gradient assembly: several in a large field, whose blocks each read
// their arguments and wait once (8192^2, three levels: 884 us with one, 765 with four, 742 with eight; 1024^2:
// 23 with one, 29 with four).
__host__ __device__ inline int fin_rounds(int64_t N1) { return N1 >= 1 << 23 ? 8 : (N1 >= 1 << 21 ? 4 : 1); }
// Fields from here on build their levels one launch each where only levels are wanted: the tiles of the
// one-pass pyramid pay for short launches (2048^2 21 us and 23, 4096^2, two levels 47 and 28).
constexpr int64_t PREP_BELOW = (int64_t)1 << 22;

// Segment of linear block b: the last segment whose blockStart <= b.
template <typename S>
__device__ __forceinline__ int find_segment(const S* __restrict__ segs, int nseg, int64_t b) {
    int lo = 0, hi = nseg - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (segs[mid].blockStart <= b) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

}  // namespace dmcr
