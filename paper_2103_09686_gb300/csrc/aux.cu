// Memory-bound kernels around the correlation: multigrid restriction / prolongation
// (Sec. 3.3), the box-penalty reduction and the loss (Sec. 3.1, Eq. L_func_dMCR), the
// fused gradient assembly + Adam update (Eq. M-update, App. B) and the counter-based
// uniform start field.  All reductions use fixed grids and fixed summation orders, so
// every result is bitwise reproducible run to run.
#include <math.h>
#include <string.h>

#include <algorithm>

#include "common.cuh"
#include "loss.cuh"

namespace dmcr {

// --------------------------------------------------------------------- multigrid

// coarse[c] = mean of the 2^d children of c (children summed in a fixed order).
__device__ __forceinline__ void restrict_one(int ndim, int64_t c0, int64_t c1, int64_t c2, const float* __restrict__ fine,
                                             float* __restrict__ coarse, int64_t i) {
    const int64_t x = i % c2, y = (i / c2) % c1, z = i / (c1 * c2);
    const int64_t f1 = 2 * c1, f2 = 2 * c2;
    float s;
    if (ndim == 2) {
        const float* r0 = fine + (2 * y) * f2 + 2 * x;
        const float* r1 = r0 + f2;
        s = ((r0[0] + r0[1]) + (r1[0] + r1[1])) * 0.25f;
    } else {
        const float* p0 = fine + ((2 * z) * f1 + 2 * y) * f2 + 2 * x;
        const float* p1 = p0 + f1 * f2;
        s = (((p0[0] + p0[1]) + (p0[f2] + p0[f2 + 1])) + ((p1[0] + p1[1]) + (p1[f2] + p1[f2 + 1]))) * 0.125f;
    }
    coarse[i] = s;
}

__global__ void restrict_kernel(const RestrictSeg* __restrict__ segs, int nseg) {
    dep_wait();
    dep_trigger();
    const int si = find_segment(segs, nseg, (int64_t)blockIdx.x);
    const RestrictSeg& sg = segs[si];
    if (sg.done != nullptr && *sg.done) return;
    const int64_t i = ((int64_t)blockIdx.x - sg.blockStart) * ELEM_TH + threadIdx.x;
    if (i >= sg.c[0] * sg.c[1] * sg.c[2]) return;
    restrict_one(sg.ndim, sg.c[0], sg.c[1], sg.c[2], sg.fine, sg.coarse, i);
}

// --------------------------------------------------------------------- pyramid

// All coarser levels of a tile in one pass over the finest field (each the mean of its 2^d
// children, summed as restrict_one does), with the tier of the values' range and the box
// excess, which need the same pass (and the phases that are bright enough for the transforms).  A
// thread reads a 2^d block; the coarser means go through shared memory.  One launch of a microsecond
// or two instead of one per level.
template <int ND>
__device__ __forceinline__ void prep_tiles(const PrepSeg& sg, int blk, float* sh, float& lo, float& hi, int& bad,
                                           int& bright, float* msh, float& e2, float& e2c) {
    constexpr int TILE = ND == 2 ? PREP_TILE2 : PREP_TILE3, H = TILE / 2;
    constexpr int CELLS = ND == 2 ? H * H : H * H * H;        // level-2 cells of a tile
    const int n0 = sg.n[0], n1 = sg.n[1], n2 = sg.n[2];
    const int64_t N = (int64_t)n0 * n1 * n2;
    const int t0 = ND == 2 ? 1 : (n0 + TILE - 1) / TILE, t1 = (n1 + TILE - 1) / TILE, t2 = (n2 + TILE - 1) / TILE;
    const int64_t tiles = (int64_t)t0 * t1 * t2 * sg.phases;
    const bool look = sg.tiers != nullptr || sg.excess != nullptr;
    // sum of the values of one phase: each warp its own share, msh[phase][warp]
    float sum = 0.f;
    int summed = 0;
    auto flush = [&]() {
        if (sg.tiers == nullptr) return;
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if ((threadIdx.x & 31) == 0) msh[summed * (ELEM_TH / 32) + (threadIdx.x >> 5)] += sum;
        sum = 0.f;
    };
    auto see = [&](float v, int ph) {
        sum += v;
        bad |= !(v == v);
        bright |= (int)(v >= SEP_WEAK) << ph;
        lo = fminf(lo, v);
        hi = fmaxf(hi, v);
        const float ex = box_excess(v);
        kahan_add(e2, e2c, ex * ex);
    };
    for (int64_t tile = blk; tile < tiles; tile += sg.nblk) {
        const int x0 = (int)(tile % t2) * TILE, y0 = (int)(tile / t2 % t1) * TILE;
        const int z0 = ND == 2 ? 0 : (int)(tile / ((int64_t)t2 * t1) % t0) * TILE;
        const int ph = (int)(tile / ((int64_t)t2 * t1 * t0));
        if (ph != summed) {
            flush();
            summed = ph;
        }
        const float* f = sg.field + ph * N;
        for (int c = threadIdx.x; c < CELLS; c += ELEM_TH) {
            const int cx = c % H, cy = c / H % H, cz = ND == 2 ? 0 : c / (H * H);
            const int x = x0 + 2 * cx, y = y0 + 2 * cy, z = z0 + 2 * cz;
            float v[ND == 2 ? 4 : 8];
#pragma unroll
            for (int k = 0; k < (ND == 2 ? 4 : 8); ++k) {
                const int xx = x + (k & 1), yy = y + (k >> 1 & 1), zz = z + (k >> 2);
                v[k] = xx < n2 && yy < n1 && zz < n0 ? f[((int64_t)zz * n1 + yy) * n2 + xx] : 0.f;
            }
            if (look) {
#pragma unroll
                for (int k = 0; k < (ND == 2 ? 4 : 8); ++k) see(v[k], ph);
            }
            if (sg.coarse == 0) continue;
            float s;
            if constexpr (ND == 2) s = ((v[0] + v[1]) + (v[2] + v[3])) * 0.25f;
            else s = (((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]))) * 0.125f;
            sh[c] = s;
            const int m1 = n1 / 2, m2 = n2 / 2, m0 = ND == 2 ? 1 : n0 / 2;
            if (x < n2 && y < n1 && z < n0)
                sg.lv[0][ph * ((int64_t)m0 * m1 * m2) + ((int64_t)(z / 2) * m1 + y / 2) * m2 + x / 2] = s;
        }
        // level l from the means of level l - 1, edge e = TILE >> l
        int src = 0, e = H;
        for (int l = 1; l < sg.coarse; ++l) {
            __syncthreads();
            const int h = e / 2, cells = ND == 2 ? h * h : h * h * h, dst = src + (ND == 2 ? e * e : e * e * e);
            const int m1 = n1 >> (l + 1), m2 = n2 >> (l + 1), m0 = ND == 2 ? 1 : n0 >> (l + 1);
            for (int c = threadIdx.x; c < cells; c += ELEM_TH) {
                const int cx = c % h, cy = c / h % h, cz = ND == 2 ? 0 : c / (h * h);
                const float* p = sh + src + (2 * cz * e + 2 * cy) * e + 2 * cx;
                float s;
                if constexpr (ND == 2) s = ((p[0] + p[1]) + (p[e] + p[e + 1])) * 0.25f;
                else
                    s = (((p[0] + p[1]) + (p[e] + p[e + 1])) +
                         ((p[e * e] + p[e * e + 1]) + (p[e * e + e] + p[e * e + e + 1]))) * 0.125f;
                sh[dst + c] = s;
                const int gx = (x0 >> (l + 1)) + cx, gy = (y0 >> (l + 1)) + cy, gz = ND == 2 ? 0 : (z0 >> (l + 1)) + cz;
                if (gx < m2 && gy < m1 && gz < m0)
                    sg.lv[l][ph * ((int64_t)m0 * m1 * m2) + ((int64_t)gz * m1 + gy) * m2 + gx] = s;
            }
            src = dst;
            e = h;
        }
        __syncthreads();
    }
    flush();
}

__global__ void __launch_bounds__(ELEM_TH) prep_kernel(const PrepSeg* __restrict__ segs, int nseg) {
    dep_wait();
    dep_trigger();
    const int si = find_segment(segs, nseg, (int64_t)blockIdx.x);
    const PrepSeg& sg = segs[si];
    if (sg.done != nullptr && *sg.done) return;
    __shared__ float sh[640];        // 2-D: 256 + 64 + 16 + 4 + 1; 3-D: 512 + 64 + 8 + 1
    __shared__ DF dsh[32];
    __shared__ int tsh[ELEM_TH / 32], bsh[ELEM_TH / 32];
    const int blk = (int)((int64_t)blockIdx.x - sg.blockStart);
    float lo = 0.f, hi = 0.f, e2 = 0.f, e2c = 0.f;
    int bad = 0, bright = 0;
    __shared__ float msh[MAX_PHASES * (ELEM_TH / 32)];
    if ((threadIdx.x & 31) == 0)
        for (int ph = 0; ph < MAX_PHASES; ++ph) msh[ph * (ELEM_TH / 32) + (threadIdx.x >> 5)] = 0.f;
    if (sg.ndim == 2) prep_tiles<2>(sg, blk, sh, lo, hi, bad, bright, msh, e2, e2c);
    else prep_tiles<3>(sg, blk, sh, lo, hi, bad, bright, msh, e2, e2c);
    if (sg.excess != nullptr) {
        const DF E = block_sum_df(df_two_sum(e2, -e2c), dsh);
        if (threadIdx.x == 0) sg.excess[blk] = make_float4(E.hi, E.lo, 0.f, 0.f);
    }
    if (sg.tiers == nullptr) return;
    if (blk == 0)
        for (int i = threadIdx.x; i < sg.nnext; i += ELEM_TH) sg.next[i] = 0;
    // the narrowest range that holds the block's values; NaN and wider fields: the direct kernels
    int t = 0;
    while (t < sg.ntier && !(lo >= sg.lo[t] && hi <= sg.hi[t])) ++t;
    if (bad || t >= sg.ntier) t = SEP_TIERS;
    t = __reduce_max_sync(0xffffffffu, t);
    bright = __reduce_or_sync(0xffffffffu, bright);
    if ((threadIdx.x & 31) == 0) tsh[threadIdx.x >> 5] = t, bsh[threadIdx.x >> 5] = bright;
    __syncthreads();
    if (threadIdx.x < sg.phases) {
        float m = 0.f;
        for (int w = 0; w < ELEM_TH / 32; ++w) m += msh[threadIdx.x * (ELEM_TH / 32) + w];
        sg.sums[blk * sg.phases + threadIdx.x] = m;
    }
    if (threadIdx.x == 0) {
        for (int w = 1; w < ELEM_TH / 32; ++w) t = max(t, tsh[w]), bright |= bsh[w];
        sg.tiers[blk] = t | bright << 8;
    }
}

void launch_prep(const PrepSeg* segs, int nseg, int64_t blocks, cudaStream_t s) {
    if (blocks <= 0) return;
    launch_dep(prep_kernel, (unsigned)blocks, ELEM_TH, 0, s, segs, nseg);
}

__global__ void restrict_plain_kernel(int ndim, int64_t c0, int64_t c1, int64_t c2, const float* __restrict__ fine,
                                      float* __restrict__ coarse) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= c0 * c1 * c2) return;
    restrict_one(ndim, c0, c1, c2, fine, coarse, i);
}

void launch_restrict(const RestrictSeg* segs, int nseg, int64_t blocks, cudaStream_t s) {
    if (blocks <= 0) return;
    launch_dep(restrict_kernel, (unsigned)blocks, ELEM_TH, 0, s, segs, nseg);
}

void launch_restrict_one(int ndim, const int64_t nf[3], const float* fine, float* coarse, cudaStream_t s) {
    const int64_t c0 = (ndim == 2) ? 1 : nf[0] / 2;
    const int64_t c1 = nf[1] / 2, c2 = nf[2] / 2;
    const int64_t Nc = c0 * c1 * c2;
    restrict_plain_kernel<<<(unsigned)((Nc + ELEM_TH - 1) / ELEM_TH), ELEM_TH, 0, s>>>(ndim, c0, c1, c2, fine, coarse);
}

// fine[f] += coarse[parent(f)] / 2^d   (transpose of restrict)   or   fine[f] = coarse[parent(f)]
__global__ void prolongate_kernel(int ndim, int64_t c0, int64_t c1, int64_t c2, const float* __restrict__ coarse,
                                  float* __restrict__ fine, int mode) {
    const int64_t f0 = (ndim == 2) ? 1 : 2 * c0, f1 = 2 * c1, f2 = 2 * c2;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= f0 * f1 * f2) return;
    const int64_t x = i % f2, y = (i / f2) % f1, z = i / (f1 * f2);
    const int64_t pz = (ndim == 2) ? 0 : z / 2;
    const float v = coarse[(pz * c1 + y / 2) * c2 + x / 2];
    if (mode == 1) fine[i] = v;
    else fine[i] += v * (ndim == 2 ? 0.25f : 0.125f);
}

void launch_prolongate(int ndim, const int64_t nc[3], const float* coarse, float* fine, int mode, cudaStream_t s) {
    const int64_t c0 = (ndim == 2) ? 1 : nc[0];
    const int64_t Nf = (ndim == 2 ? 4 : 8) * c0 * nc[1] * nc[2];
    const int th = 256;
    prolongate_kernel<<<(unsigned)((Nf + th - 1) / th), th, 0, s>>>(ndim, c0, nc[1], nc[2], coarse, fine, mode);
}

// --------------------------------------------------------------------- loss

__device__ __forceinline__ double block_sum_d(double v, double* sh) {
    // fixed-order tree over the block (blockDim.x a power of two <= 1024)
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    const double r = sh[0];
    __syncthreads();
    return r;
}

// Loss of the instances whose descriptor kernels do not finish it (three-point and corrected
// descriptors, FFT levels), grid (max nblk, instances): double-float partial sums over the
// instance's own nblk blocks (a fixed grid per problem size) -- sum (D - D_des)^2 and
// sum D_des^2 over the descriptor, and sum ex^2 of the box excess over the field (when the
// penalty is on); its last block sums the partials in a fixed order and finishes the loss
// (a launch of its own: 9 us more).
__global__ void __launch_bounds__(256, 5) stats_kernel(const PenSeg* __restrict__ segs) {
    dep_wait();
    dep_trigger();
    const PenSeg& sg = segs[blockIdx.y];
    if (sg.done != nullptr && *sg.done) return;
    if ((int)blockIdx.x >= sg.nblk) return;
    __shared__ DF sh[3 * 8];
    const int64_t stride = (int64_t)sg.nblk * blockDim.x;
    const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    // per-thread compensated (Kahan) FP32 sums in a fixed order -- FP64 arithmetic is slow on
    // this part and a thread sums only about 8 terms (stats_blocks) -- then a double-float
    // (two-sum) tree across the block
    float r2 = 0.f, r2c = 0.f, t2 = 0.f, t2c = 0.f, e2 = 0.f, e2c = 0.f;
    // the terms of this thread in order, their loads issued eight at a time, the last ones too
    // (terms past the end are zeros: one by one they took as long as all the others)
    constexpr int U = 8;
    for (int64_t k = i0; k < sg.K; k += U * stride) {
        float tv[U], dv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool in = k + u * stride < sg.K;
            tv[u] = in ? sg.target[k + u * stride] : 0.f;
            dv[u] = in ? sg.desc[k + u * stride] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float r = dv[u] - tv[u];
            kahan_add(r2, r2c, r * r);
            kahan_add(t2, t2c, tv[u] * tv[u]);
        }
    }
    if (sg.field != nullptr) {
        for (int64_t i = i0; i < sg.N; i += U * stride) {
            float fv[U];
#pragma unroll
            for (int u = 0; u < U; ++u) fv[u] = i + u * stride < sg.N ? sg.field[i + u * stride] : 0.f;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const float e = box_excess(fv[u]);
                kahan_add(e2, e2c, e * e);
            }
        }
    }
    // Kahan's (sum, comp) stands for sum - comp
    DF v[3] = {df_two_sum(r2, -r2c), df_two_sum(t2, -t2c), df_two_sum(e2, -e2c)};
    block_sums_df(v, sh);
    if (threadIdx.x == 0) {
        sg.sums[blockIdx.x] = make_float4(v[0].hi, v[0].lo, v[1].hi, v[1].lo);
        sg.excess[blockIdx.x] = make_float4(v[2].hi, v[2].lo, 0.f, 0.f);
    }
    loss_arrive(*sg.loss, sg.nblk, sh);
}

void launch_penalty(const PenSeg* segs, int nseg, int maxblk, cudaStream_t s) {
    if (nseg <= 0) return;
    launch_dep(stats_kernel, dim3(maxblk, nseg), 256, 0, s, segs);
}

// blocks of the loss statistics: about 2048 terms per block, 256 .. NPEN_BLOCKS, a power of two
int stats_blocks(int64_t K, int64_t N) {
    const int64_t work = K > N ? K : N;
    int b = 256;
    while (b < NPEN_BLOCKS && (int64_t)b * 2048 < work) b *= 2;
    return b;
}

// Corrected two-point descriptor, forward: map every block in place (entry 0 is read, never
// written, so the map needs no second buffer).
__global__ void tilde_map_kernel(const TildeSeg* __restrict__ segs, int nseg) {
    dep_wait();
    dep_trigger();
    const int si = find_segment(segs, nseg, (int64_t)blockIdx.x);
    const TildeSeg& sg = segs[si];
    if (sg.done != nullptr && *sg.done) return;
    const int64_t k = ((int64_t)blockIdx.x - sg.blockStart) * ELEM_TH + threadIdx.x;
    if (k < 1 || k >= sg.K) return;
    sg.desc[k] = (sg.desc[k] - sg.q * sg.desc[0]) / (1.f - sg.q);
}

void launch_tilde_map(const TildeSeg* segs, int nseg, int64_t blocks, cudaStream_t s) {
    if (blocks <= 0) return;
    launch_dep(tilde_map_kernel, (unsigned)blocks, ELEM_TH, 0, s, segs, nseg);
}

// Corrected two-point descriptor, backward: one block per segment, sum_{k >= 1} (src - sub)
// in FP64 in a fixed order.
__global__ void tilde_sum_kernel(const TildeSeg* __restrict__ segs) {
    dep_wait();
    dep_trigger();
    const TildeSeg& sg = segs[blockIdx.x];
    if (sg.done != nullptr && *sg.done) return;
    __shared__ double sh[256];
    double acc = 0.0;
    for (int64_t k = 1 + threadIdx.x; k < sg.K; k += blockDim.x)
        acc += (double)sg.src[k] - (sg.sub != nullptr ? (double)sg.sub[k] : 0.0);
    acc = block_sum_d(acc, sh);
    if (threadIdx.x == 0) *sg.tsum = (float)acc;
}

void launch_tilde_sum(const TildeSeg* segs, int nseg, cudaStream_t s) {
    if (nseg <= 0) return;
    launch_dep(tilde_sum_kernel, nseg, 256, 0, s, segs);
}

// --------------------------------------------------------------------- gradient + Adam

// g(y) = sum_l 2^{-d(l-1)} sum_chunks part_l[chunk][ancestor_l(y)]  (+ penalty gradient),
// then either written out, or used for one Adam step (Keras form) on the field.  Position i's
// chunk sums for the chunks c = q (mod SUB) of every level, each level's chunks in order,
// their loads issued eight at a time.
template <int SUB>
__device__ __forceinline__ float chunk_sums(const FinalArgs& a, int64_t i, int q) {
    // coordinates only where a coarser level needs them, in 32 bits where they fit (the 64-bit
    // divisions: 22 us for 128^3, one level, 9 so)
    int64_t x = i, y = 0, z = 0;
    if (a.levels > 1) {
        if (a.n1[0] * a.n1[1] * a.n1[2] <= 0x7fffffff) {
            const unsigned n2 = (unsigned)a.n1[2], n1 = (unsigned)a.n1[1], row = (unsigned)i / n2;
            x = (unsigned)i - row * n2;
            z = row / n1;
            y = row - (unsigned)z * n1;
        } else {
            x = i % a.n1[2];
            y = (i / a.n1[2]) % a.n1[1];
            z = i / (a.n1[1] * a.n1[2]);
        }
    }
    float g = 0.f, scale = 1.f;
    const float step = a.ndim == 2 ? 0.25f : 0.125f;
    const bool sep = a.tier != nullptr && *a.tier < SEP_TIERS;
    for (int l = 0; l < a.levels; ++l) {
        const int64_t lz = a.ndim == 2 ? 0 : (z >> l);
        const int64_t li = l == 0 ? i : (lz * a.nl[l][1] + (y >> l)) * a.nl[l][2] + (x >> l);
        const int64_t jump = SUB * a.Nl[l];
        const float* p = (sep ? a.sparts[l] : a.parts[l]) + li + q * a.Nl[l];
        const int nc = sep ? 1 : a.nChunks[l];
        float s = 0.f;
        int c = q;
        for (; c + 7 * SUB < nc; c += 8 * SUB) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u, p += jump) v[u] = *p;
#pragma unroll
            for (int u = 0; u < 8; ++u) s += v[u];
        }
        for (; c < nc; c += SUB, p += jump) s += *p;
        g = fmaf(scale, s, g);
        scale *= step;
    }
    return g;
}

// A block covers ELEM_TH / SUB positions with SUB threads each.  SUB = 1 (a large field):
// one thread per position, a warp reads 32 consecutive positions of a chunk.  SUB = FIN_SUB
// (a small field: few positions for many chunk partials): thread (q, p) -- q = threadIdx.x /
// positions, so a warp still reads consecutive positions of one chunk -- sums the chunks
// c = q (mod FIN_SUB) and the FIN_SUB partials are added in a fixed order through shared
// memory.
// The segment's arguments (written at least two launches earlier) and the field and moments at
// the thread's position are read before the adjoint kernels' end is waited for.
template <int SUB>
__global__ void __launch_bounds__(ELEM_TH) final_kernel(const FinalSeg* __restrict__ segs, int nseg) {
    constexpr int NPOS = ELEM_TH / SUB;
    __shared__ FinalSeg sg;
    static_assert(sizeof(FinalSeg) % 4 == 0 && sizeof(FinalSeg) / 4 <= ELEM_TH, "one word a thread");
    const FinalSeg* src = segs + find_segment(segs, nseg, (int64_t)blockIdx.x);
    if (threadIdx.x < sizeof(FinalSeg) / 4)
        reinterpret_cast<uint32_t*>(&sg)[threadIdx.x] = reinterpret_cast<const uint32_t*>(src)[threadIdx.x];
    __syncthreads();
    const FinalArgs& a = sg.a;
    const int64_t N1 = a.n1[0] * a.n1[1] * a.n1[2];
    const int q = threadIdx.x / NPOS, pl = threadIdx.x % NPOS;
    const int rounds = SUB == 1 ? fin_rounds(N1) : 1;
    int64_t i = ((int64_t)blockIdx.x - sg.blockStart) * NPOS * rounds + pl;
    float M = 0.f, m0 = 0.f, v0 = 0.f;
    auto load = [&]() {
        if (i >= N1 || q != 0) return;
        if (a.M != nullptr) {
            M = a.M[i];
            m0 = a.m[i];
            v0 = a.v[i];
        } else if (a.sc != nullptr && a.field != nullptr) {
            M = a.field[i];
        }
    };
    load();
    dep_wait();
    dep_trigger();
    if (sg.done != nullptr && *sg.done) return;
    for (int r = 0;;) {
        float g = i < N1 ? chunk_sums<SUB>(a, i, q) : 0.f;
        if constexpr (SUB > 1) {
            __shared__ float part[SUB][NPOS];
            part[q][pl] = g;
            __syncthreads();
            if (q != 0) return;
            for (int u = 1; u < SUB; ++u) g += part[u][pl];
        }
        if (i >= N1) return;
        if (a.sc != nullptr && a.field != nullptr) {
            const float f = a.M != nullptr && a.M != a.field ? a.field[i] : M;
            const float ex = box_excess(f);
            const float dex = f > 1.f ? 1.f : (f < 0.f ? -1.f : 0.f);
            g = fmaf(a.sc->pen_coef * ex, dex, g);
        }
        if (a.grad_out != nullptr) a.grad_out[i] = g;
        if (a.M != nullptr) {
            const float m = fmaf(a.beta1, m0, (1.f - a.beta1) * g);
            const float v = fmaf(a.beta2, v0, (1.f - a.beta2) * g * g);
            a.m[i] = m;
            a.v[i] = v;
            a.M[i] = M - a.sc->lr_t * m / (sqrtf(v) + a.eps);
        }
        if (++r >= rounds) return;
        i += NPOS;
        load();
    }
}

void launch_final(const FinalSeg* segs, int nseg, int64_t blocks, int sub, cudaStream_t s) {
    if (blocks <= 0) return;
    if (sub == 1)
        launch_dep(final_kernel<1>, (unsigned)blocks, ELEM_TH, 0, s, segs, nseg);
    else
        launch_dep(final_kernel<FIN_SUB>, (unsigned)blocks, ELEM_TH, 0, s, segs, nseg);
}

// Writes up to BLOB_BYTES of host data, passed by value as a kernel parameter, to device
// memory: stream ordered, no host synchronisation, and valid inside a graph capture.  Different
// lanes read different parameter words, which the constant path serves one address at a time:
// 16 bytes a thread and a warp per block keep that serial chain short (15 KB: 6.0 -> 2.3 us).
// The parameters are copied whole at every launch, so they come in sizes: the host spends 25 us on
// the descriptor of a 32^2 field (2 KB), 28 with 30 KB.
constexpr int BLOB_BYTES = 30720;
template <int BYTES>
struct Blob {
    unsigned int quads;
    uint4 data[BYTES / 16];
};

template <int BYTES>
__global__ void __launch_bounds__(32) blob_kernel(const __grid_constant__ Blob<BYTES> b, uint4* __restrict__ dst) {
    dep_wait();
    dep_trigger();
    const unsigned int i = blockIdx.x * 32 + threadIdx.x;
    if (i < b.quads) dst[i] = b.data[i];
}

namespace {
template <int BYTES>
void blob_part(const unsigned char* src, size_t n, unsigned char* dst, cudaStream_t s) {
    static thread_local Blob<BYTES> b;
    const size_t quads = (n + 15) / 16;
    if (n % 16) memset(&b.data[quads - 1], 0, 16);
    memcpy(b.data, src, n);
    b.quads = (unsigned int)quads;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((quads + 31) / 32));
    cfg.blockDim = dim3(32);
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    // by pointer: the parameters are copied once, by the launch
    uint4* out = reinterpret_cast<uint4*>(dst);
    void* args[] = {&b, &out};
    cudaLaunchKernelExC(&cfg, reinterpret_cast<const void*>(blob_kernel<BYTES>), args);
}
}  // namespace

void launch_blob(const void* host, size_t bytes, void* dst, cudaStream_t s) {
    const unsigned char* src = static_cast<const unsigned char*>(host);
    unsigned char* out = static_cast<unsigned char*>(dst);
    for (size_t off = 0; off < bytes;) {
        const size_t n = std::min<size_t>(bytes - off, BLOB_BYTES);
        if (n <= 2048) blob_part<2048>(src + off, n, out + off, s);
        else if (n <= 4096) blob_part<4096>(src + off, n, out + off, s);
        else if (n <= 10240) blob_part<10240>(src + off, n, out + off, s);
        else blob_part<BLOB_BYTES>(src + off, n, out + off, s);
        off += (n + 15) / 16 * 16;
    }
}

// --------------------------------------------------------------------- start field

// SplitMix64 (Steele, Lea & Flood 2014): state seed + (i+1) * golden gamma, then the
// published three-step mix; value = top 24 bits * 2^-24.
__global__ void init_uniform_kernel(float* __restrict__ f, int64_t count, uint64_t seed) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    uint64_t z = seed + (uint64_t)(i + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z = z ^ (z >> 31);
    f[i] = (float)(z >> 40) * (1.0f / 16777216.0f);
}

void launch_init_uniform(float* field, int64_t count, uint64_t seed, cudaStream_t s) {
    const int th = 256;
    init_uniform_kernel<<<(unsigned)((count + th - 1) / th), th, 0, s>>>(field, count, seed);
}

// The rounded field used to evaluate a reconstruction (Sec. 4.1): values >= 1/2 become
// phase 1, the rest phase 0.
__global__ void round_field_kernel(const float* __restrict__ src, float* __restrict__ dst, int64_t count) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    dst[i] = src[i] >= 0.5f ? 1.f : 0.f;
}

void launch_round_field(const float* src, float* dst, int64_t count, cudaStream_t s) {
    if (count <= 0) return;
    const int th = 256;
    round_field_kernel<<<(unsigned)((count + th - 1) / th), th, 0, s>>>(src, dst, count);
}

}  // namespace dmcr
