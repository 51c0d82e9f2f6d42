// Separable evaluation of the soft-thresholded two-point descriptor and its adjoint
// (sm_103a).  Paper: arXiv 2103.09686, Sec. 3.2.2-3.2.4 and the gradient of Sec. 3.1/3.3.
//
// The pair function F(u, v) = f((u + v) / 2)^2 is smooth on the bounded range of a relaxed
// field, so around a value c it is, to FP32 accuracy, a short sum over features that vanish at c:
//     F(u, v) = F(u, c) + F(c, v) - F(c, c) + sum_k s_k q_k(u) q_k(v),  s_k = +-1,
//     q_k(u) = p_k(u) - p_k(c), p_k piecewise polynomials (sep_basis.cpp, built on the host in FP64),
// 14 terms on [-1/16, 17/16] at alpha = 10.  c is the mean of the field, or 0 for a field whose
// mean lies near 0: what most pairs of a field consist of is then evaluated directly, not as a
// difference of features rounded to FP32.  The descriptor is a mean and a sum of autocorrelations of
// R feature fields, and the gradient a sum of convolutions of the same features with the window
// coefficients G:
//     S(r) = (2/N) sum_x F(M_x, c) - F(c, c) + (1/N) sum_k s_k sum_x q_k(M_x) q_k(M_{x+r}),
//     g(y) = F_u(M_y, c) sum_r G(r) + sum_k s_k p_k'(M_y) sum_r G(r) q_k(M_{y+r}).
// (Several phases: a value each, F(M^a, c_b) and F(c_a, M^b).)
// Both are diagonal in Fourier space: the work per position falls from the window's K pair
// evaluations (8321 at +-64) to R transforms (5 R log2 N operations).  Features of equal sign
// are packed in pairs, z = p_1 + i p_2: Re IDFT(|Z|^2) = autocorr(p_1) + autocorr(p_2), and a
// real even G acts on both parts at once, so no mirrored frequency is ever read.
//
//   prep_kernel (aux.cu) the tier (basis) that covers the field's values; none: the direct kernels run
//   sep_feat    features of whole rows + transform along x             -> Z; sums of F(M, c)
//   sep_fft_y   3-D: transform along y, in place
//   sep_power   last axis: transform, sum_k s_k conj(Z^a_k) Z^b_k, inverse along the same
//               axis, cropped to the window; the mean of F(M, c) joins the frequency 0
//   sep_inv_y   3-D: inverse along y, cropped to the window
//   sep_desc    inverse along x, cropped to the window: the descriptor
//   sep_gx/gy   the window's coefficients G embedded and transformed along x (and y)
//   sep_mul     last axis: transform of G, then per feature pair transform, product, inverse; sum of G
//   sep_grad    inverse along x, sum_k s_k p_k'(M_y) Q_k(y) and the term of F_u(M, c): the gradient
//
// The power of the frequency 0, the features' means, is summed in FP64 with the mean of F(M, c) and
// added after the inverse transform, so the FP32 transforms only carry fluctuations.  Fixed grids and orders: results are bitwise reproducible.
#include <math.h>

#include <algorithm>
#include <mutex>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "loss.cuh"

namespace dmcr {

// ------------------------------------------------------------------------- coefficients (host)

// Coefficients in device memory: the first SEP_SLOTS_DEV alphas a process uses get a slot of a
// static array, filled once per device by a synchronous copy on a stream of its own (also while
// another stream is being captured); slots are never rewritten, so kernels and graphs may keep
// reading them.  Null when there is no slot: the call uploads the coefficients with its tables.
namespace {
constexpr int SEP_SLOTS_DEV = 8, SEP_SLOT_LEN = 32768;
__device__ float2 g_sep_coef[SEP_SLOTS_DEV][SEP_SLOT_LEN];
}  // namespace

const float2* sep_device_coef(const SepBasis& b) {
    struct Slot {
        int dev;
        float alpha;
        const float2* ptr;
    };
    static std::mutex mu;
    static std::vector<Slot>* slots = new std::vector<Slot>();
    if (b.coef.size() > (size_t)SEP_SLOT_LEN) return nullptr;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    std::lock_guard<std::mutex> lk(mu);
    int used = 0;
    for (const Slot& s : *slots)
        if (s.dev == dev) {
            if (s.alpha == b.alpha) return s.ptr;
            ++used;
        }
    if (used >= SEP_SLOTS_DEV) return nullptr;
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    if (cudaThreadExchangeStreamCaptureMode(&mode) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    void* base = nullptr;
    cudaStream_t s = nullptr;
    bool ok = cudaGetSymbolAddress(&base, g_sep_coef) == cudaSuccess &&
              cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) == cudaSuccess;
    float2* dst = static_cast<float2*>(base) + (size_t)used * SEP_SLOT_LEN;
    ok = ok && cudaMemcpyAsync(dst, b.coef.data(), b.coef.size() * sizeof(SepCoef), cudaMemcpyHostToDevice, s) == cudaSuccess;
    if (s) ok = cudaStreamSynchronize(s) == cudaSuccess && ok;
    if (s) cudaStreamDestroy(s);
    cudaThreadExchangeStreamCaptureMode(&mode);
    if (!ok) {
        cudaGetLastError();
        return nullptr;
    }
    slots->push_back({dev, b.alpha, dst});
    return dst;
}

// ------------------------------------------------------------------------- plan (host)

// Transform lengths: any n <= SEP_MAX_N; radices 8, 4, 2, 3, 5, 7, then the remaining primes
// (a direct sum over the prime, O(p) per point).
bool sep_axis(int64_t n, SepAxis& ax) {
    if (n < 1 || n > SEP_MAX_N) return false;
    ax.n = (int)n;
    ax.nrad = 0;
    ax.fast = 0;
    for (int k = 4; (1 << k) <= SEP_MAX_N; ++k)
        if (n == (1 << k)) ax.fast = k;
    int m = (int)n;
    auto put = [&](int r) {
        if (ax.nrad >= SEP_MAX_RAD) return false;
        ax.rad[ax.nrad++] = (unsigned short)r;
        m /= r;
        return true;
    };
    while (m % 8 == 0)
        if (!put(8)) return false;
    for (int r : {4, 2, 3, 5, 7})
        while (m % r == 0)
            if (!put(r)) return false;
    for (int r = 11; m > 1; r += 2)
        while (m % r == 0)
            if (!put(r)) return false;
    return true;
}

// Estimated seconds per point and axis of a loss and gradient with 7 feature pairs: powers of
// two, and the general stages (primes by their length).
double sep_axis_cost(const SepAxis& ax) {
    if (ax.fast) return 1.3e-10;
    double c = 0.0;
    for (int i = 0; i < ax.nrad; ++i) c += ax.rad[i] <= 8 ? 1e-10 : 3e-11 * ax.rad[i];
    return c;
}

namespace {
int pow2_floor(int v) {
    int p = 1;
    while (2 * p <= v) p *= 2;
    return p;
}
}  // namespace

// Adjacent columns of a strided axis per block.  A block holds SEP_BLOCK_PTS points of a power
// of two: its remaining factor goes to feature pairs (or planes).  3-D grids take 16 columns
// (128-byte lines).  2-D grids trade the width of their segments against the number of blocks:
// 8 columns (64 bytes) where those fill the device -- long columns, several phases -- and 4
// otherwise (256^2: sep_power 16.7 us with 4, 20.6 us with 8; nine phase pairs of 512^2: 213 and
// 148 us; two columns, half a sector, took 43 us where four took 31).
int sep_cols(const SepAxis& ax, bool wide, int phases) {
    const int n = ax.n;
    if (ax.fast) {
        const int lines = SEP_BLOCK_PTS / n;
        const int narrow = std::max(n >= 512 || phases > 1 ? 8 : 4, lines / 8);   // at most 8 pairs side by side
        return std::min(std::min(lines, 16), wide ? 16 : narrow);
    }
    if (n > 1024) return 2;
    return std::max(4, std::min(16, pow2_floor(2048 / n)));
}

// Rows per block of the window kernels.
int sep_window_rows(const SepAxis& ax) {
    const int pts = ax.fast ? SEP_BLOCK_PTS : 2048;
    return std::max(1, std::min(ax.fast ? 64 : 16, pow2_floor(std::max(1, pts / ax.n))));
}

// Rows per block of the feature and gradient kernels, of a grid with `rows` rows.  A block
// holds 2048 points (SEP_SLOTS pairs of as many rows as fit, or a share of the pairs of one
// row); large grids take several such groups one after another, up to 8, as long as about
// 1200 blocks (two per resident one) remain: start-up (tables, twiddles) is paid once.
int sep_feature_rows(const SepAxis& ax, int64_t rows) {
    const int base = std::max(1, std::min(16, pow2_floor(std::max(1, 2048 / (ax.n * SEP_SLOTS)))));
    if (!ax.fast) return base;
    int loops = 1;
    while (loops < 8 && rows / (base * loops * 2) >= 1216) loops *= 2;
    return base * loops;
}

// ------------------------------------------------------------------------- transforms (device)

namespace {

__device__ __forceinline__ float2 cmulf(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// packed sums and differences: one issue slot for both parts (a - b as an exact FMA with -1)
__device__ __forceinline__ float2 caddf(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 csubf(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 swapf(float2 a) { return make_float2(a.y, a.x); }
// times -i
__device__ __forceinline__ float2 rot(float2 a) { return make_float2(a.y, -a.x); }

// Only forward transforms are written: an inverse exchanges real and imaginary parts of its
// input and output.

// Lines live in shared memory with one pad element (8 bytes) after every 16: the radix-8
// stages' strided writes then spread over the banks.
__device__ __forceinline__ int spad(int i) { return i + (i >> 4); }

// tw[t] = exp(-2 pi i t / n), from sincospi of an argument reduced to an eighth of a turn
__device__ __forceinline__ void fill_twiddles(float2* tw, int n) {
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
        // angle = 2 pi t / n = (pi / 4)(o + r / n); odd octants are reflected about pi / 4
        const int o = 8 * t / n;
        int r = 8 * t - o * n;
        const bool flip = o & 1;
        if (flip) r = n - r;
        float s, c;
        sincospif((float)r / (float)(4 * n), &s, &c);
        if (flip) { const float x = s; s = c; c = x; }
        const int quad = o >> 1;
        const float cs = quad == 0 ? c : (quad == 1 ? -s : (quad == 2 ? -c : s));
        const float sn = quad == 0 ? s : (quad == 1 ? c : (quad == 2 ? -s : -c));
        tw[t] = make_float2(cs, -sn);
    }
}

__device__ __forceinline__ void bfly4(float2& a, float2& b, float2& c, float2& d) {
    const float2 s0 = caddf(a, c), d0 = csubf(a, c), s1 = caddf(b, d), t = csubf(b, d);
    a = caddf(s0, s1);
    b = make_float2(d0.x + t.y, d0.y - t.x);
    c = csubf(s0, s1);
    d = make_float2(d0.x - t.y, d0.y + t.x);
}

// V[q] = sum_r v[r] exp(-2 pi i r q / R) in place
template <int R>
__device__ __forceinline__ void butterfly(float2 (&v)[R]) {
    if constexpr (R == 2) {
        const float2 t = csubf(v[0], v[1]);
        v[0] = caddf(v[0], v[1]);
        v[1] = t;
    } else if constexpr (R == 4) {
        bfly4(v[0], v[1], v[2], v[3]);
    } else if constexpr (R == 8) {
        // even and odd halves, then the eighth roots
        bfly4(v[0], v[2], v[4], v[6]);
        bfly4(v[1], v[3], v[5], v[7]);
        constexpr float h = 0.70710678118654752440f;
        const float2 hp = make_float2(h, h), hm = make_float2(-h, -h);
        const float2 w1 = make_float2(v[3].x + v[3].y, v[3].y - v[3].x);     // odd 1 times (1 - i)
        const float2 w3 = make_float2(v[7].y - v[7].x, -v[7].x - v[7].y);    // odd 3 times -(1 + i)
        const float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o2 = v[5];
        v[0] = caddf(e0, o0);
        v[4] = csubf(e0, o0);
        v[1] = __ffma2_rn(w1, hp, e1);
        v[5] = __ffma2_rn(w1, hm, e1);
        v[2] = make_float2(e2.x + o2.y, e2.y - o2.x);
        v[6] = make_float2(e2.x - o2.y, e2.y + o2.x);
        v[3] = __ffma2_rn(w3, hp, e3);
        v[7] = __ffma2_rn(w3, hm, e3);
    } else {
        // odd radices: pair r with R - r; the cosines and sines of 2 pi j / R are constants
        constexpr int H = (R - 1) / 2;
        constexpr float C3[1] = {-0.5f}, S3[1] = {0.86602540378443864676f};
        constexpr float C5[2] = {0.30901699437494742410f, -0.80901699437494742410f},
                        S5[2] = {0.95105651629515357212f, 0.58778525229247312917f};
        constexpr float C7[3] = {0.62348980185873353053f, -0.22252093395631440429f, -0.90096886790241912624f},
                        S7[3] = {0.78183148246802980871f, 0.97492791218182360702f, 0.43388373911755812048f};
        float2 p[H], m[H];
#pragma unroll
        for (int r = 0; r < H; ++r) {
            p[r] = caddf(v[r + 1], v[R - 1 - r]);
            m[r] = rot(csubf(v[r + 1], v[R - 1 - r]));
        }
        const float2 v0 = v[0];
#pragma unroll
        for (int r = 0; r < H; ++r) v[0] = caddf(v[0], p[r]);
#pragma unroll
        for (int q = 1; q <= H; ++q) {
            float2 a = v0, b = make_float2(0.f, 0.f);
#pragma unroll
            for (int r = 1; r <= H; ++r) {
                const int j = (r * q) % R, jj = j <= H ? j : R - j;      // angle index, folded
                const float c = R == 3 ? C3[jj - 1] : (R == 5 ? C5[jj - 1 < 2 ? jj - 1 : 0] : C7[jj - 1]);
                const float s0 = R == 3 ? S3[jj - 1] : (R == 5 ? S5[jj - 1 < 2 ? jj - 1 : 0] : S7[jj - 1]);
                const float s = j <= H ? s0 : -s0;
                a = make_float2(fmaf(c, p[r - 1].x, a.x), fmaf(c, p[r - 1].y, a.y));
                b = make_float2(fmaf(s, m[r - 1].x, b.x), fmaf(s, m[r - 1].y, b.y));
            }
            v[q] = caddf(a, b);
            v[R - q] = csubf(a, b);
        }
    }
}

// ---- powers of two: 8 points per thread in registers
//
// T = N / 8 threads hold a line; thread t holds the points t + e T (e = 0 .. 7) before the
// first stage and after the last, so that a product between two transforms needs no exchange.
// Stockham stages of radix 8 (the last one 2 or 4), exchanged through shared memory in two
// alternating buffers: one barrier per exchange.
template <int N>
struct Line {
    float2* buf[2];           // this line in the two buffers
    const float2* tw;
    int t;
};

// WARP: the line's threads are consecutive lanes of one warp
template <bool WARP>
__device__ __forceinline__ void line_sync() {
    if (WARP) __syncwarp();
    else __syncthreads();
}

// Hides a value from the optimiser: a loop over rounds recomputes the few addresses derived from
// it instead of keeping dozens of them in registers (the column kernels spilled 800 bytes).
__device__ __forceinline__ int opaque(int v) {
    asm volatile("" : "+r"(v));
    return v;
}
template <int N>
__device__ __forceinline__ Line<N> opaque(Line<N> ln) {
    ln.t = opaque(ln.t);
    return ln;
}

template <int N, int Ns, bool WARP, int PAR>
__device__ __forceinline__ void p2_stages(float2 (&v)[8], const Line<N>& ln) {
    constexpr int T = N / 8, REM = N / Ns, R = REM >= 8 ? 8 : REM, M = 8 / R;
#pragma unroll
    for (int m = 0; m < M; ++m) {
        const int k = (ln.t + m * T) & (Ns - 1);
        float2 u[R];
#pragma unroll
        for (int r = 0; r < R; ++r) u[r] = v[m + r * M];
        if (Ns > 1) {
#pragma unroll
            for (int r = 1; r < R; ++r) u[r] = cmulf(u[r], ln.tw[k * r * (REM / R)]);
        }
        butterfly<R>(u);
#pragma unroll
        for (int r = 0; r < R; ++r) v[m + r * M] = u[r];
    }
    if constexpr (Ns * R < N) {
        static_assert(R == 8, "only the last stage has another radix");
        float2* b = ln.buf[PAR];
        // point (t - k) 8 + k + q Ns of the next stage's input; the pads are constants of q
        const int k = ln.t & (Ns - 1), o = (ln.t - k) * 8 + k;
        float2* out = b + spad(o);
#pragma unroll
        for (int q = 0; q < 8; ++q) out[q * Ns + (Ns == 1 ? 0 : (Ns == 8 ? q / 2 : q * Ns / 16))] = v[q];
        line_sync<WARP>();
        const float2* in = b + spad(ln.t);
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = in[e * T + (T >= 16 ? e * T / 16 : (e * T) / 16)];
        p2_stages<N, Ns * R, WARP, PAR ^ 1>(v, ln);
    }
}

// exchanges of one transform (the buffer parity the next one starts with)
__host__ __device__ constexpr int p2_exchanges(int N) { return N <= 8 ? 0 : (N <= 64 ? 1 : (N <= 512 ? 2 : 3)); }

template <int N, bool WARP, int PAR>
__device__ __forceinline__ void p2_fft(float2 (&v)[8], const Line<N>& ln) {
    p2_stages<N, 1, WARP, PAR>(v, ln);
}

__device__ __forceinline__ void swap8(float2 (&v)[8]) {
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = swapf(v[e]);
}

// line pitch (float2 elements) of rows: consecutive lines start 2 T banks apart
template <int N>
__host__ __device__ constexpr int row_pitch() {
    int p = N - 1 + (N - 1) / 16 + 1;
    const int want = N >= 128 ? 0 : N / 8;
    while (p % 16 != want) ++p;
    return p;
}

// ---- any other length: stages over lines in shared memory

// t / d for 0 <= t < 2^20 through a float reciprocal: (t + 1/2) / d is at least 1/(2 d) away
// from an integer, and the rounding of the product is below t 2^-22 / d
__device__ __forceinline__ int fdiv(int t, float inv) { return (int)(((float)t + 0.5f) * inv); }

// One Stockham stage of radix R over `lines` lines (pitch elements apart) src -> dst.
template <int R>
__device__ __forceinline__ void sep_stage(const float2* __restrict__ src, float2* __restrict__ dst,
                                          const float2* __restrict__ tw, int n, int lines, int pitch, int Ns) {
    const int nR = n / R;
    const int tstep = nR / Ns;
    const float inv_nR = 1.0f / (float)nR, inv_Ns = 1.0f / (float)Ns;
    for (int t = threadIdx.x; t < lines * nR; t += blockDim.x) {
        const int l = fdiv(t, inv_nR), j = t - l * nR;
        const int blk = fdiv(j, inv_Ns), k = j - blk * Ns;
        const float2* in = src + l * pitch;
        float2 v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = in[spad(j + r * nR)];
        if (Ns > 1) {
#pragma unroll
            for (int r = 1; r < R; ++r) v[r] = cmulf(v[r], tw[k * r * tstep]);
        }
        butterfly<R>(v);
        float2* out = dst + l * pitch;
        const int o = blk * Ns * R + k;
#pragma unroll
        for (int q = 0; q < R; ++q) out[spad(o + q * Ns)] = v[q];
    }
}

// A prime radix p > 7: one thread per output, a direct sum over the p inputs.
__device__ __forceinline__ void sep_stage_prime(const float2* __restrict__ src, float2* __restrict__ dst,
                                                const float2* __restrict__ tw, int n, int lines, int pitch, int Ns,
                                                int p) {
    const int np = n / p, tstep = np / Ns;
    const float inv_n = 1.0f / (float)n, inv_np = 1.0f / (float)np, inv_Ns = 1.0f / (float)Ns;
    for (int t = threadIdx.x; t < lines * n; t += blockDim.x) {
        const int l = fdiv(t, inv_n), e = t - l * n;
        const int q = fdiv(e, inv_np), j = e - q * np;
        const int blk = fdiv(j, inv_Ns), k = j - blk * Ns;
        const float2* in = src + l * pitch;
        const int step = k * tstep + q * np;      // < n: the angle of one input to the next
        float2 a = in[spad(j)];
        int w = 0, at = j;
        for (int r = 1; r < p; ++r) {
            w += step;
            if (w >= n) w -= n;
            at += np;
            const float2 c = tw[w], x = in[spad(at)];
            a.x = fmaf(x.x, c.x, fmaf(-x.y, c.y, a.x));
            a.y = fmaf(x.x, c.y, fmaf(x.y, c.x, a.y));
        }
        dst[l * pitch + spad(blk * Ns * p + k + q * Ns)] = a;
    }
}

// Forward transform of `lines` lines in shared memory: from `a`, through `b` and back; returns
// the buffer that holds the result.  Begins and ends with a barrier.  One copy of the code
// serves every call.
__device__ __noinline__ float2* transform(const SepAxis& ax, float2* a, float2* b, const float2* tw, int lines,
                                          int pitch) {
    int Ns = 1;
    __syncthreads();
    for (int s = 0; s < ax.nrad; ++s) {
        const int R = ax.rad[s];
        switch (R) {
            case 8: sep_stage<8>(a, b, tw, ax.n, lines, pitch, Ns); break;
            case 4: sep_stage<4>(a, b, tw, ax.n, lines, pitch, Ns); break;
            case 2: sep_stage<2>(a, b, tw, ax.n, lines, pitch, Ns); break;
            case 3: sep_stage<3>(a, b, tw, ax.n, lines, pitch, Ns); break;
            case 5: sep_stage<5>(a, b, tw, ax.n, lines, pitch, Ns); break;
            case 7: sep_stage<7>(a, b, tw, ax.n, lines, pitch, Ns); break;
            default: sep_stage_prime(a, b, tw, ax.n, lines, pitch, Ns, R); break;
        }
        Ns *= R;
        float2* x = a;
        a = b;
        b = x;
        __syncthreads();
    }
    return a;
}

// ---- what a block works on

extern __shared__ __align__(16) float2 sep_smem[];

// Dynamic shared memory: twiddles of the axis, then two buffers of whole lines.
struct SepShared {
    float2 *tw, *a, *b;
};
__device__ __forceinline__ SepShared sep_shared(float2* sm, int n, int lines, int pitch) {
    SepShared s;
    s.tw = sm;
    s.a = sm + ((n + 1) & ~1);
    s.b = s.a + lines * pitch;
    return s;
}

struct SepBlock {
    SepLevel lv;
    int a, b, block, part, parts, tier;      // block: group of lines; part of parts: its share of the pairs
};

// Before the wait for the predecessor: finds the block's item (every thread looks at one),
// copies its level to shared memory (tables are written at least two launches earlier) and
// fills the twiddles of `axis(level)`.  After it: reads the instance's tier and returns false
// when there is nothing to do -- the instance has stopped, or (TIERED) its field needs the
// direct kernels.
template <bool TIERED, typename AXIS>
__device__ __forceinline__ bool enter(const SepTables& tb, const SepItem* __restrict__ items, int nitem,
                                      SepBlock& bk, float2* tw, AXIS axis) {
    int count = 0;
    for (int base = 0; base < nitem; base += blockDim.x) {
        const int i = base + threadIdx.x;
        count += __syncthreads_count(i < nitem && items[i].blockStart <= (int64_t)blockIdx.x);
    }
    const SepItem& it = items[count - 1];
    const uint32_t* src = reinterpret_cast<const uint32_t*>(tb.level + it.level);
    uint32_t* dst = reinterpret_cast<uint32_t*>(&bk.lv);
    for (int i = threadIdx.x; i < (int)(sizeof(SepLevel) / 4); i += blockDim.x) dst[i] = src[i];
    if (threadIdx.x == 0) {
        bk.a = it.a;
        bk.b = it.b;
        const int local = (int)((int64_t)blockIdx.x - it.blockStart);
        bk.block = local / it.parts;
        bk.part = local - bk.block * it.parts;
        bk.parts = it.parts;
    }
    const int *tier = it.tier, *done = it.done;
    __syncthreads();
    fill_twiddles(tw, axis(bk.lv));
    dep_wait();
    dep_trigger();
    const bool stopped = done != nullptr && *done;
    const int t = TIERED ? *tier : 0;
    if (threadIdx.x == 0) bk.tier = t;
    __syncthreads();
    return !stopped && t < SEP_TIERS;
}

__device__ __forceinline__ int axis_x(const SepLevel& lv) { return lv.n2; }
__device__ __forceinline__ int axis_y(const SepLevel& lv) { return lv.n1; }
__device__ __forceinline__ int axis_last(const SepLevel& lv) { return lv.n0 > 1 ? lv.n0 : lv.n1; }

// runs body(std::integral_constant<int, N>) for the power of two N = 2^k, 16 <= N <= 2048
template <typename F>
__device__ __forceinline__ void for_pow2(int k, F&& body) {
    switch (k) {
        case 4: body(std::integral_constant<int, 16>()); break;
        case 5: body(std::integral_constant<int, 32>()); break;
        case 6: body(std::integral_constant<int, 64>()); break;
        case 7: body(std::integral_constant<int, 128>()); break;
        case 8: body(std::integral_constant<int, 256>()); break;
        case 9: body(std::integral_constant<int, 512>()); break;
        case 10: body(std::integral_constant<int, 1024>()); break;
        default: body(std::integral_constant<int, 2048>()); break;
    }
}

}  // namespace

// ------------------------------------------------------------------------- features

namespace {

// C values M of one line: their segments (offsets into the coefficient tables) and positions
// u = SEP_SEG M - k in them, both exact.
template <int C>
__device__ __forceinline__ void locate(const SepTier& t, const float (&M)[C], int (&seg)[C], float (&u)[C]) {
#pragma unroll
    for (int e = 0; e < C; ++e) {
        const float y = (float)SEP_SEG * M[e];
        seg[e] = min(max(__float2int_rn(y) - t.seg0, 0), t.nseg - 1);
        u[e] = y - (float)(seg[e] + t.seg0);
    }
}

// One packed pair of features (DERIV: of their derivatives) at C located values: a polynomial
// of nc coefficients per value, the coefficients of its segment gathered from global memory
// (`cf`: those of the pair; step: from one power to the next).  The tables of a tier stay in
// L1, a gather touches one or two lines, and the cost does not grow with the range.  Against
// one Chebyshev series over the whole range (35 .. 127 terms) this takes 8 gathers and 7 FFMA2
// per pair: the row kernels' instructions per point fell from 156 to about 75.
template <bool DERIV, int C>
__device__ __forceinline__ void eval_features(const float2* __restrict__ cf, int step, int nc, const int (&seg)[C],
                                              const float (&u)[C], float2 (&out)[C]) {
    const float2* c = cf + (nc - 1) * step;
#pragma unroll
    for (int e = 0; e < C; ++e) {
        out[e] = __ldg(c + seg[e]);
        if (DERIV) out[e] = __fmul2_rn(out[e], make_float2((float)(nc - 1), (float)(nc - 1)));
    }
    for (int j = nc - 2; j >= (DERIV ? 1 : 0); --j) {
        c -= step;
        const float2 f = make_float2((float)j, (float)j);
#pragma unroll
        for (int e = 0; e < C; ++e) {
            float2 k = __ldg(c + seg[e]);
            if (DERIV) k = __fmul2_rn(k, f);
            out[e] = __ffma2_rn(out[e], make_float2(u[e], u[e]), k);
        }
    }
}

// F(M, c) and its derivative by M.  z = exp((alpha / 2)(1.5 - c - M)) is
// wanted to 1e-7 of itself: c is a multiple of 2^-10, so 1.5 - c is exact, and the exponent keeps its
// rounding errors.  (Beyond exp(80) f is its limit.)
__device__ __forceinline__ float pair_with(const SepTables& tb, float M, float c, float& slope) {
    const float h = 0.5f * tb.alpha;
    const DF d = df_two_sum(1.5f - c, -M);
    const float e = fminf(h * d.hi, 80.f), low = e < 80.f ? fmaf(h, d.lo, fmaf(h, d.hi, -e)) : 0.f;
    float z = expf(e);
    z = fmaf(z, low, z);
    const float s = __fdividef(1.f, 1.f + z), f = fmaf(tb.c1, s, tb.c3);       // 1 + z < 2^126
    slope = f * (tb.c1 * tb.alpha * s) * (z * s);
    return f * f;
}
__device__ __forceinline__ float pair_with(const SepTables& tb, float M, float c) {
    float slope;
    return pair_with(tb, M, c, slope);
}

// rows of a block of the feature and gradient kernels: SLOTS feature pairs side by side
template <int N>
struct RowShape {
    static constexpr int T = N / 8, LINES = SEP_ROW_THREADS / T;
    static constexpr int SLOTS = LINES < SEP_SLOTS ? LINES : SEP_SLOTS;
    static constexpr int ROWS = LINES / SLOTS;
    static constexpr bool WARP = T <= 32;
};

template <int N>
__device__ __forceinline__ Line<N> row_line(float2* sm, int line, int t, int lines) {
    constexpr int P = row_pitch<N>();
    Line<N> ln;
    ln.tw = sm;
    ln.buf[0] = sm + N + line * P;
    ln.buf[1] = ln.buf[0] + lines * P;
    ln.t = t;
    return ln;
}

}  // namespace

// item: (level, phase a); blocks: groups of rows.  Features of whole rows and their transform
// along x, and the warps' sums of F(M, c).  Every block combines the range blocks' tiers and sums;
// the first block of the finest level leaves the tier and c for the later kernels.  Bound by
// latency (coefficient gathers from L1, exchanges): it issues 35 % of the time.  Seven pairs:
// 512^2, three levels 27 us; 1024^2, five levels 86 us; 128^3, two levels 97 us, 8 % of it for the
// features' offsets and F(M, c) (one series over the whole range instead of local polynomials:
// twice the instructions).
__global__ void __launch_bounds__(SEP_ROW_THREADS, 4) sep_feat_kernel(const __grid_constant__ SepTables tb,
                                                                      const SepItem* __restrict__ items, int nitem) {
    __shared__ SepBlock bk;
    constexpr int NW = SEP_ROW_THREADS / 32;
    __shared__ int tsh[NW], bsh[NW];
    __shared__ float csh[MAX_PHASES][NW];
    __shared__ float2 offset[SEP_MAX_PAIRS];      // p_k(c)
    if (!enter<false>(tb, items, nitem, bk, sep_smem, axis_x)) return;
    const SepLevel& lv = bk.lv;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    {
        int t = 0, bright = 0;
        for (int i = threadIdx.x; i < lv.ntiers; i += blockDim.x) {
            t = max(t, lv.tiers[i] & 0xff);
            bright |= lv.tiers[i] >> 8;
        }
        for (int ph = 0; ph < lv.phases; ++ph) {
            float m = 0.f;
            for (int i = threadIdx.x; i < lv.ntiers; i += blockDim.x) m += lv.msum[i * lv.phases + ph];
            for (int o = 16; o > 0; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
            if (lane == 0) csh[ph][warp] = m;
        }
        t = __reduce_max_sync(0xffffffffu, t);
        bright = __reduce_or_sync(0xffffffffu, bright);
        if (lane == 0) tsh[warp] = t, bsh[warp] = bright;
    }
    float2* sm = sep_smem;
    const int rowsN = lv.n0 * lv.n1, n = lv.n2;
    __syncthreads();
    int tier = tsh[0], bright = bsh[0];
    for (int i = 1; i < NW; ++i) tier = max(tier, tsh[i]), bright |= bsh[i];
    if (bright != (1 << lv.phases) - 1) tier = SEP_TIERS;      // a phase without a value of SEP_WEAK
    // the values c: the means on a grid of 2^-10, 0 for those in the segment around 0 (where the
    // features of the background are exactly 0 already)
    auto center = [&](int ph) {
        float m = 0.f;
        for (int i = 0; i < NW; ++i) m += csh[ph][i];
        m *= lv.invN1;
        return m > 0.5f / SEP_SEG ? rintf(1024.f * m) * (1.f / 1024.f) : 0.f;
    };
    if (lv.first && bk.a == 0 && bk.block == 0 && threadIdx.x < lv.phases) lv.center[threadIdx.x] = center(threadIdx.x);
    if (lv.first && bk.a == 0 && bk.block == 0 && threadIdx.x == 0) *lv.tier = tier;
    if (tier >= SEP_TIERS) return;
    const SepTier& t = tb.tier[tier];
    const float2* __restrict__ cf = tb.coef + t.coef;
    const int step = t.npair * t.nseg;
    const int row0 = bk.block * lv.rowsF, rows = min(lv.rowsF, rowsN - row0);
    const float* __restrict__ field = lv.field + (int64_t)bk.a * lv.N + (int64_t)row0 * n;
    float2* __restrict__ Z = lv.Z + (int64_t)bk.a * lv.maxPairs * lv.N + (int64_t)row0 * n;
    const float own = center(bk.a);
    if (threadIdx.x < t.npair) {
        const float x[1] = {own};
        float u[1];
        int seg[1];
        float2 f[1];
        locate<1>(t, x, seg, u);
        eval_features<false, 1>(cf + threadIdx.x * t.nseg, step, t.nc, seg, u, f);
        offset[threadIdx.x] = f[0];
    }
    if (lv.phi != nullptr)
        for (int b = 0; b < lv.phases; ++b) {
            const float c = center(b);
            float s = 0.f;
            for (int e = threadIdx.x; e < rows * n; e += blockDim.x) s += pair_with(tb, field[e], c);
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) lv.phi[(int64_t)(bk.a * lv.phases + b) * lv.nphi + bk.block * NW + warp] = s;
        }
    __syncthreads();
    if (lv.ax[2].fast) {
        for_pow2(lv.ax[2].fast, [&](auto c) {
            constexpr int N = decltype(c)::value;
            using S = RowShape<N>;
            const int line = threadIdx.x / S::T, p = line % S::SLOTS;
            const Line<N> ln = row_line<N>(sm, line, threadIdx.x % S::T, S::LINES);
            for (int row = line / S::SLOTS; row < lv.rowsF; row += S::ROWS) {
                const bool in = row < rows;
                float x[8], u[8];
                int seg[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) x[e] = in ? field[row * N + ln.t + e * S::T] : 0.f;
                locate<8>(t, x, seg, u);
                for (int p0 = 0; p0 < t.npair; p0 += S::SLOTS) {
                    const bool live = in && p0 + p < t.npair;
                    float2 v[8];
                    if (live) {
                        eval_features<false, 8>(cf + (p0 + p) * t.nseg, step, t.nc, seg, u, v);
                        const float2 c = offset[p0 + p];
#pragma unroll
                        for (int e = 0; e < 8; ++e) v[e] = csubf(v[e], c);
                    }
                    p2_fft<N, S::WARP, 0>(v, opaque(ln));
                    if (live) {
                        float2* out = Z + (int64_t)(p0 + p) * lv.N + row * N + ln.t;
#pragma unroll
                        for (int e = 0; e < 8; ++e) out[e * S::T] = v[e];
                    }
                    // the next round starts in the buffer this one started in
                    if (p2_exchanges(N) & 1) line_sync<S::WARP>();
                }
            }
        });
        return;
    }
    const int pitch = spad(n - 1) + 2;
    const float inv_n = 1.0f / (float)n;
    const SepShared s = sep_shared(sm, n, lv.rowsF * SEP_SLOTS, pitch);
    for (int p0 = 0; p0 < t.npair; p0 += SEP_SLOTS) {
        const int nc = min(SEP_SLOTS, t.npair - p0);
        __syncthreads();
        for (int e = threadIdx.x; e < rows * nc * n; e += blockDim.x) {
            const int q = fdiv(e, inv_n), i = e - q * n;        // q = l nc + c
            const int l = q / nc, c = q - l * nc;
            const float x[1] = {field[l * n + i]};
            float u[1];
            int seg[1];
            locate<1>(t, x, seg, u);
            float2 f[1];
            eval_features<false, 1>(cf + (p0 + c) * t.nseg, step, t.nc, seg, u, f);
            s.a[q * pitch + spad(i)] = csubf(f[0], offset[p0 + c]);
        }
        const float2* r = transform(lv.ax[2], s.a, s.b, s.tw, rows * nc, pitch);
        for (int e = threadIdx.x; e < rows * nc * n; e += blockDim.x) {
            const int q = fdiv(e, inv_n), i = e - q * n;
            const int l = q / nc, c = q - l * nc;
            Z[(int64_t)(p0 + c) * lv.N + l * n + i] = r[q * pitch + spad(i)];
        }
    }
}

// ------------------------------------------------------------------------- columns

namespace {

// Threads of a block over L adjacent columns (fastest, for coalesced rows), T per line and the
// SLOTS = SEP_THREADS / (L T) groups side by side (feature pairs, or planes).
template <int N>
struct Cols {
    static constexpr int T = N / 8;
    int L, l, slot, slots;
    Line<N> ln;
    __device__ __forceinline__ explicit Cols(int L_) : L(L_) {
        const int sh = 31 - __clz(L);
        l = threadIdx.x & (L - 1);
        const int r = threadIdx.x >> sh;
        ln.t = r % T;
        slot = r / T;
        slots = SEP_THREADS / T >> sh;
        const int pitch = sep_pitch(N, L);
        ln.tw = sep_smem;
        ln.buf[0] = sep_smem + N + (slot * L + l) * pitch;
        ln.buf[1] = ln.buf[0] + slots * L * pitch;
    }
};

// the columns of one block along a strided axis
struct ColGroup {
    int n, L, cols;
    int64_t base, stride;      // first element of the group within one grid; step along the axis
};

// last axis: z in 3-D, y in 2-D
__device__ __forceinline__ ColGroup last_axis(const SepLevel& lv, int block, int& x0, int& y) {
    ColGroup g;
    g.L = lv.colsL;
    const int xg = (lv.n2 + g.L - 1) / g.L;
    x0 = (block % xg) * g.L;
    y = lv.n0 > 1 ? block / xg : 0;
    g.n = lv.n0 > 1 ? lv.n0 : lv.n1;
    g.cols = min(g.L, lv.n2 - x0);
    g.stride = lv.n0 > 1 ? (int64_t)lv.n1 * lv.n2 : lv.n2;
    g.base = (int64_t)y * lv.n2 + x0;
    return g;
}

__device__ __forceinline__ const SepAxis& last_ax(const SepLevel& lv) { return lv.n0 > 1 ? lv.ax[0] : lv.ax[1]; }

// A thread's eight points of one grid.  Element offsets within a grid fit 32 bits (at most
// SEP_MAX_POINTS points).
template <int N>
__device__ __forceinline__ void load8(const float2* __restrict__ src, const ColGroup& g, const Cols<N>& c, bool on,
                                      float2 (&v)[8]) {
    const int stride = opaque((int)g.stride), step = (N / 8) * stride;
    const float2* p = src + (int)g.base + (c.ln.t * stride + c.l);
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = on && c.l < g.cols ? p[e * step] : make_float2(0.f, 0.f);
}

template <int N>
__device__ __forceinline__ void store8(float2* __restrict__ dst, const ColGroup& g, const Cols<N>& c, bool on,
                                       const float2 (&v)[8]) {
    const int stride = opaque((int)g.stride), step = (N / 8) * stride;
    float2* p = dst + (int)g.base + (c.ln.t * stride + c.l);
    if (on && c.l < g.cols) {
#pragma unroll
        for (int e = 0; e < 8; ++e) p[e * step] = v[e];
    }
}

// columns into shared lines (any length)
__device__ __forceinline__ void load_cols(const float2* __restrict__ src, const ColGroup& g, int pitch, float2* dst) {
    const int sh = 31 - __clz(g.L);
    for (int e = threadIdx.x; e < g.L * g.n; e += blockDim.x) {
        const int l = e & (g.L - 1), i = e >> sh;
        dst[l * pitch + spad(i)] = l < g.cols ? src[g.base + i * g.stride + l] : make_float2(0.f, 0.f);
    }
}

}  // namespace

// Middle axis of 3-D, in place on Z (forward) or on the product spectra (INVERSE).  item:
// (level, phase a); blocks: groups of planes' columns (x fastest, then z).  A block walks the
// feature pairs, loading the next pair's columns while it transforms the current ones (128^3, two
// levels, seven pairs: 53 us; a block for every pair: 99).
template <bool INVERSE>
__global__ void __launch_bounds__(SEP_THREADS, 2) sep_fft_y_kernel(const __grid_constant__ SepTables tb,
                                                                   const SepItem* __restrict__ items, int nitem) {
    __shared__ SepBlock bk;
    if (!enter<true>(tb, items, nitem, bk, sep_smem, axis_y)) return;
    const SepLevel& lv = bk.lv;
    float2* sm = sep_smem;
    const int L = lv.colsY, n = lv.n1;
    const int xg = (lv.n2 + L - 1) / L, groups = xg * lv.n0;
    const int slots = lv.ax[1].fast ? SEP_BLOCK_PTS / (L * n) : 1;
    const int g0 = bk.block * slots, npair = tb.tier[bk.tier].npair;
    float2* grid = (INVERSE ? lv.Q : lv.Z) + (int64_t)bk.a * lv.maxPairs * lv.N;
    auto group = [&](int gi) {
        ColGroup g;
        g.n = n;
        g.L = L;
        const int x0 = (gi % xg) * L, z = gi / xg;
        g.cols = min(L, lv.n2 - x0);
        g.stride = lv.n2;
        g.base = (int64_t)z * lv.n1 * lv.n2 + x0;
        return g;
    };
    if (lv.ax[1].fast) {
        for_pow2(lv.ax[1].fast, [&](auto cc) {
            constexpr int N = decltype(cc)::value;
            const Cols<N> c(L);
            const bool on = g0 + c.slot < groups;
            const ColGroup g = group(on ? g0 + c.slot : 0);
            float2 nx[8];
            load8<N>(grid, g, c, on, nx);
            for (int p = 0; p < npair; ++p) {
                float2 v[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = INVERSE ? swapf(nx[e]) : nx[e];
                if (p + 1 < npair) load8<N>(grid + (int64_t)(p + 1) * lv.N, g, c, on, nx);
                p2_fft<N, false, 0>(v, opaque(c.ln));
                if (p2_exchanges(N) & 1) __syncthreads();
                if (INVERSE) swap8(v);
                store8<N>(grid + (int64_t)p * lv.N, g, c, on, v);
            }
        });
        return;
    }
    const ColGroup g = group(g0);
    const int pitch = sep_pitch(n, L), sh = 31 - __clz(L);
    const SepShared s = sep_shared(sm, n, L, pitch);
    for (int p = 0; p < npair; ++p, grid += lv.N) {
        __syncthreads();
        for (int e = threadIdx.x; e < L * n; e += blockDim.x) {
            const int l = e & (L - 1), i = e >> sh;
            const float2 v = l < g.cols ? grid[g.base + i * g.stride + l] : make_float2(0.f, 0.f);
            s.a[l * pitch + spad(i)] = INVERSE ? swapf(v) : v;
        }
        const float2* r = transform(lv.ax[1], s.a, s.b, s.tw, L, pitch);
        for (int e = threadIdx.x; e < L * n; e += blockDim.x) {
            const int l = e & (L - 1), i = e >> sh;
            const float2 v = r[l * pitch + spad(i)];
            if (l < g.cols) grid[g.base + i * g.stride + l] = INVERSE ? swapf(v) : v;
        }
    }
}

// ------------------------------------------------------------------------- last axis: power

namespace {
// FP64 value as an FP32 pair
__device__ __forceinline__ float2 split(double v) {
    const float hi = (float)v;
    return make_float2(hi, (float)(v - (double)hi));
}
}  // namespace

// item: (level, phases a, b).  Sums s_k conj(Z^a_k) Z^b_k over the feature pairs and writes the
// inverse along the last axis, cropped to r = 0 .. P (-r belongs to the pair (b, a)).  The block that
// holds the frequency 0 adds the means of F(M, c) there.  CROSS: a and b may differ.  Bound by latency: one or two blocks an SM.  512^2, three levels, seven pairs:
// 27 us with two shares of the pairs at the finest level (33 with one); 128^3, two levels: 101 us;
// nine phase pairs of 512^2: 153 us.
template <bool CROSS>
__global__ void __launch_bounds__(SEP_THREADS, CROSS ? 1 : 2)
sep_power_kernel(const __grid_constant__ SepTables tb, const SepItem* __restrict__ items, int nitem) {
    __shared__ SepBlock bk;
    __shared__ double dcs[SEP_THREADS / 2];
    __shared__ DF psh[SEP_THREADS / 32];  // sum F(M^a, c_b) + sum F(c_a, M^b), one share a warp
    if (!enter<true>(tb, items, nitem, bk, sep_smem, axis_last)) return;
    const SepLevel& lv = bk.lv;
    float2* sm = sep_smem;
    const SepTier& t = tb.tier[bk.tier];
    int x0, y;
    const ColGroup g = last_axis(lv, bk.block, x0, y);
    const SepAxis& ax = last_ax(lv);
    const bool dc_block = x0 == 0 && y == 0;
    const float2* Za = lv.Z + (int64_t)bk.a * lv.maxPairs * lv.N;
    const float2* Zb = lv.Z + (int64_t)bk.b * lv.maxPairs * lv.N;
    float2* Zw = lv.Z;                       // one phase: the spectra are left for sep_mul
    const int pair = bk.a * lv.phases + bk.b;
    const int P = lv.n0 > 1 ? lv.P0 : lv.P1;
    // 3-D: U[r][y][x]; 2-D: V[r][x]
    float2* out = (lv.n0 > 1 ? lv.U : lv.V) + (int64_t)(pair + bk.part) * (lv.n0 > 1 ? lv.strideU : lv.strideV) + g.base;
    const bool cross = CROSS && bk.a != bk.b;
    if (dc_block && bk.part == 0) {
        DF v{0.f, 0.f};
        const float* pa = lv.phi + (int64_t)(bk.a * lv.phases + bk.b) * lv.nphi;
        const float* pb = lv.phi + (int64_t)(bk.b * lv.phases + bk.a) * lv.nphi;
        for (int i = threadIdx.x; i < lv.nphi; i += blockDim.x) v = df_add(v, df_two_sum(pa[i], pb[i]));
        for (int o = 16; o > 0; o >>= 1)
            v = df_add(v, DF{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)});
        if ((threadIdx.x & 31) == 0) psh[threadIdx.x >> 5] = v;
    }
    // by the thread that holds the frequency 0, a barrier or more later
    auto means = [&]() {
        DF v = psh[0];
        for (int w = 1; w < SEP_THREADS / 32; ++w) v = df_add(v, psh[w]);
        const double twice = (double)pair_with(tb, lv.center[bk.a], lv.center[bk.b]);
        return (double)lv.N * (((double)v.hi + (double)v.lo) - (double)lv.N * twice);
    };
    if (ax.fast) {
        for_pow2(ax.fast, [&](auto cc) {
            constexpr int N = decltype(cc)::value, T = N / 8;
            constexpr int PAR1 = p2_exchanges(N) & 1;
            const Cols<N> c(g.L);
            // one phase: the eight sums of a thread wait in shared memory (its own words), which
            // keeps the transform's 64 registers free of spills
            float* own = reinterpret_cast<float*>(sm + N + 2 * c.slots * c.L * sep_pitch(N, c.L)) + threadIdx.x;
            float2 acc[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                if (CROSS) acc[e] = make_float2(0.f, 0.f);
                else own[e * SEP_THREADS] = 0.f;
            }
            double dc = 0.0;
            const bool has_dc = dc_block && c.l == 0 && c.ln.t == 0;
            for (int p0 = bk.part * c.slots; p0 < t.npair; p0 += bk.parts * c.slots) {
                const int p = p0 + c.slot;
                const float sg = p < t.npos ? 1.f : -1.f;
                float2 v[8];
                load8<N>(Za + (int64_t)p * lv.N, g, c, p < t.npair, v);
                if (!CROSS) {
                    p2_fft<N, false, 0>(v, opaque(c.ln));
                    if (PAR1 != 0) __syncthreads();   // the next round starts in buffer 0 again
                    if (lv.keep) store8<N>(Zw + (int64_t)p * lv.N, g, c, p < t.npair, v);
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        own[e * SEP_THREADS] = fmaf(sg, fmaf(v[e].x, v[e].x, v[e].y * v[e].y), own[e * SEP_THREADS]);
                    if (has_dc) dc += (double)sg * ((double)v[0].x * v[0].x + (double)v[0].y * v[0].y);
                } else if (!cross) {
                    p2_fft<N, false, 0>(v, opaque(c.ln));
                    if (PAR1 != 0) __syncthreads();
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        acc[e].x = fmaf(sg, __fadd_rn(__fmul_rn(v[e].x, v[e].x), __fmul_rn(v[e].y, v[e].y)), acc[e].x);
                    if (has_dc) dc += (double)sg * ((double)v[0].x * v[0].x + (double)v[0].y * v[0].y);
                } else {
                    float2 u[8];
                    load8<N>(Zb + (int64_t)p * lv.N, g, c, p < t.npair, u);
                    p2_fft<N, false, 0>(v, opaque(c.ln));
                    if (PAR1 != 0) __syncthreads();
                    p2_fft<N, false, 0>(u, opaque(c.ln));
                    if (PAR1 != 0) __syncthreads();
                    // conj(v) u; the imaginary part as a difference of rounded products, so that
                    // exchanging a and b gives exactly the conjugate
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        acc[e].x = fmaf(sg, __fadd_rn(__fmul_rn(v[e].x, u[e].x), __fmul_rn(v[e].y, u[e].y)), acc[e].x);
                        acc[e].y = fmaf(sg, __fsub_rn(__fmul_rn(v[e].x, u[e].y), __fmul_rn(v[e].y, u[e].x)), acc[e].y);
                    }
                    if (has_dc) dc += (double)sg * ((double)v[0].x * u[0].x + (double)v[0].y * u[0].y);
                }
            }
            if (!CROSS) {
#pragma unroll
                for (int e = 0; e < 8; ++e) acc[e] = make_float2(own[e * SEP_THREADS], 0.f);
            }
            // sum over the slots in a fixed order; the mean's power goes on in FP64
            if (has_dc) dcs[c.slot] = dc;
            __syncthreads();
            if (c.slots > 1) {
                float2* red = sep_smem + N;
#pragma unroll
                for (int e = 0; e < 8; ++e) red[e * SEP_THREADS + threadIdx.x] = acc[e];
                __syncthreads();
                const int group = SEP_THREADS / c.slots, at = threadIdx.x % group;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    float2 s = red[e * SEP_THREADS + at];
                    for (int k = 1; k < c.slots; ++k) s = caddf(s, red[e * SEP_THREADS + at + k * group]);
                    acc[e] = s;
                }
                __syncthreads();
            }
            if (has_dc && c.slot == 0) {
                double s = dcs[0];
                for (int k = 1; k < c.slots; ++k) s += dcs[k];
                if (bk.part == 0) s += means();
                lv.dc[pair + bk.part] = split(s * lv.scaleD);
            }
            if (has_dc) acc[0] = make_float2(0.f, 0.f);
            swap8(acc);
            p2_fft<N, false, 0>(acc, opaque(c.ln));
            if (c.slot == 0 && c.l < g.cols) {
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int i = c.ln.t + e * T;
                    if (i <= P) out[i * g.stride + c.l] = swapf(acc[e]);
                }
            }
        });
        return;
    }
    const int pitch = sep_pitch(g.n, g.L), sh = 31 - __clz(g.L), total = g.L * g.n;
    const SepShared s = sep_shared(sm, g.n, g.L, pitch);
    float2 acc[SEP_OWN], za[SEP_OWN];
#pragma unroll
    for (int q = 0; q < SEP_OWN; ++q) acc[q] = make_float2(0.f, 0.f);
    double dc = 0.0;
    const bool has_dc = dc_block && threadIdx.x == 0;   // element 0 is frequency 0
    auto own = [&](auto f) {
#pragma unroll
        for (int q = 0; q < SEP_OWN; ++q) {
            const int e = threadIdx.x + q * SEP_THREADS;
            if (e < total) f(q, (e & (g.L - 1)) * pitch + spad(e >> sh));
        }
    };
    for (int p = bk.part; p < t.npair; p += bk.parts) {
        const float sg = p < t.npos ? 1.f : -1.f;
        __syncthreads();
        load_cols(Za + (int64_t)p * lv.N, g, pitch, s.a);
        const float2* r = transform(ax, s.a, s.b, s.tw, g.L, pitch);
        if (cross) {
            own([&](int q, int at) { za[q] = r[at]; });
            __syncthreads();
            load_cols(Zb + (int64_t)p * lv.N, g, pitch, s.a);
            r = transform(ax, s.a, s.b, s.tw, g.L, pitch);
        }
        if (lv.keep && !CROSS)
            for (int e = threadIdx.x; e < total; e += blockDim.x) {
                const int l = e & (g.L - 1), i = e >> sh;
                if (l < g.cols) Zw[(int64_t)p * lv.N + g.base + i * g.stride + l] = r[l * pitch + spad(i)];
            }
        own([&](int q, int at) {
            const float2 v = r[at], u = cross ? za[q] : v;
            acc[q].x = fmaf(sg, __fadd_rn(__fmul_rn(u.x, v.x), __fmul_rn(u.y, v.y)), acc[q].x);
            acc[q].y = fmaf(sg, __fsub_rn(__fmul_rn(u.x, v.y), __fmul_rn(u.y, v.x)), acc[q].y);
            if (q == 0 && has_dc) dc += (double)sg * ((double)u.x * v.x + (double)u.y * v.y);
        });
    }
    if (has_dc) {
        if (bk.part == 0) dc += means();
        lv.dc[pair + bk.part] = split(dc * lv.scaleD);
        acc[0] = make_float2(0.f, 0.f);
    }
    __syncthreads();
    own([&](int q, int at) { s.a[at] = swapf(acc[q]); });
    const float2* r = transform(ax, s.a, s.b, s.tw, g.L, pitch);
    for (int e = threadIdx.x; e < g.L * (P + 1); e += blockDim.x) {
        const int l = e & (g.L - 1), i = e >> sh;
        if (l < g.cols) out[i * g.stride + l] = swapf(r[l * pitch + spad(i)]);
    }
}

// ------------------------------------------------------------------------- 3-D middle axis of the window

// item: (level, phases a, b); blocks: groups of columns (x fastest, then kept rz).  DESC: U -> V,
// inverse along y cropped to -P1 .. P1.  Otherwise V -> U: G's rows embedded along y and
// transformed.
template <bool DESC>
__global__ void __launch_bounds__(SEP_THREADS, 2) sep_win_y_kernel(const __grid_constant__ SepTables tb,
                                                                   const SepItem* __restrict__ items, int nitem) {
    __shared__ SepBlock bk;
    if (!enter<true>(tb, items, nitem, bk, sep_smem, axis_y)) return;
    const SepLevel& lv = bk.lv;
    float2* sm = sep_smem;
    const int L = lv.colsY, n = lv.n1, P1 = lv.P1, wy = 2 * P1 + 1;
    const int xg = (lv.n2 + L - 1) / L, groups = xg * (lv.P0 + 1);
    const int slots = lv.ax[1].fast ? SEP_BLOCK_PTS / (L * n) : 1;
    const int pair = bk.a * lv.phases + bk.b;
    float2* U = lv.U + (int64_t)pair * lv.strideU;
    float2* V = lv.V + (int64_t)pair * lv.strideV;
    auto window = [&](const float2* src, int i, int64_t stride) {
        // ry = i and ry = i - n (both at the aliased ry = +-n/2)
        float2 v = make_float2(0.f, 0.f);
        if (i <= P1) v = src[(int64_t)(i + P1) * stride];
        if (i > 0 && n - i <= P1) v = caddf(v, src[(int64_t)(i - n + P1) * stride]);
        return v;
    };
    if (lv.ax[1].fast) {
        for_pow2(lv.ax[1].fast, [&](auto cc) {
            constexpr int N = decltype(cc)::value, T = N / 8;
            const Cols<N> c(L);
            const int gi = bk.block * slots + c.slot, k = gi / xg, x = (gi % xg) * L + c.l;
            const bool on = gi < groups && x < lv.n2;
            float2* u = U + (int64_t)k * lv.n1 * lv.n2 + x;
            float2* w = V + (int64_t)k * wy * lv.n2 + x;
            float2 v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int i = c.ln.t + e * T;
                v[e] = !on ? make_float2(0.f, 0.f) : (DESC ? swapf(u[(int64_t)i * lv.n2]) : window(w, i, lv.n2));
            }
            p2_fft<N, false, 0>(v, opaque(c.ln));
            if (!on) return;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int i = c.ln.t + e * T;
                if (!DESC) {
                    u[(int64_t)i * lv.n2] = v[e];
                } else {
                    if (i <= P1) w[(int64_t)(i + P1) * lv.n2] = swapf(v[e]);
                    if (i > 0 && N - i <= P1) w[(int64_t)(i - N + P1) * lv.n2] = swapf(v[e]);
                }
            }
        });
        return;
    }
    const int gi = bk.block, k = gi / xg, x0 = (gi % xg) * L, cols = min(L, lv.n2 - x0);
    const int pitch = sep_pitch(n, L), sh = 31 - __clz(L);
    const SepShared s = sep_shared(sm, n, L, pitch);
    U += (int64_t)k * lv.n1 * lv.n2 + x0;
    V += (int64_t)k * wy * lv.n2 + x0;
    for (int e = threadIdx.x; e < L * n; e += blockDim.x) {
        const int l = e & (L - 1), i = e >> sh;
        float2 v = make_float2(0.f, 0.f);
        if (l < cols) v = DESC ? swapf(U[(int64_t)i * lv.n2 + l]) : window(V + l, i, lv.n2);
        s.a[l * pitch + spad(i)] = v;
    }
    const float2* r = transform(lv.ax[1], s.a, s.b, s.tw, L, pitch);
    for (int e = threadIdx.x; e < L * (DESC ? wy : n); e += blockDim.x) {
        const int l = e & (L - 1), i = e >> sh;
        if (l >= cols) continue;
        if (DESC) {
            const int ry = i - P1;
            V[(int64_t)i * lv.n2 + l] = swapf(r[l * pitch + spad(ry < 0 ? ry + n : ry)]);
        } else {
            U[(int64_t)i * lv.n2 + l] = r[l * pitch + spad(i)];
        }
    }
}

// ------------------------------------------------------------------------- window rows

namespace {

// row `row` of the kept half of the window -> (rz, ry): 3-D rz = 0 .. P0 and every ry, 2-D
// ry = 0 .. P1
__device__ __forceinline__ void window_row(const SepLevel& lv, int row, int& rz, int& ry) {
    if (lv.n0 > 1) {
        const int wy = 2 * lv.P1 + 1;
        rz = row / wy;
        ry = row - rz * wy - lv.P1;
    } else {
        rz = 0;
        ry = row;
    }
}

__device__ __forceinline__ int window_rows(const SepLevel& lv) {
    return lv.n0 > 1 ? (lv.P0 + 1) * (2 * lv.P1 + 1) : lv.P1 + 1;
}

// Canonical half-window index of (rz, ry, rx), -1 if it is not in the half window.
__device__ __forceinline__ int half_index(const SepLevel& lv, int rz, int ry, int rx) {
    const int Px = lv.P2, Py = lv.P1;
    if (rz == 0 && ry == 0) return rx >= 0 ? rx : -1;
    if (rz == 0) return ry > 0 ? (Px + 1) + (ry - 1) * (2 * Px + 1) + (rx + Px) : -1;
    if (rz < 0) return -1;
    return (Px + 1) + Py * (2 * Px + 1) + ((rz - 1) * (2 * Py + 1) + (ry + Py)) * (2 * Px + 1) + (rx + Px);
}

}  // namespace

// item: (level, phases a, b); blocks: groups of rowsW window rows.  Inverse along x: the
// entries of block (a, b); with a loss to evaluate, its share of the loss' sums too.  With
// lv.fuse (one phase, a loss and its gradient in one call) a row goes straight on: its residuals
// D - D_des are G up to the loss' factor gscale, which sep_mul applies, so they are embedded and
// transformed here (the rows of sep_gx).  17 blocks at 512^2: 20 us, the chain of one row's two
// transforms, the descriptor and the loss (a launch of sep_gx less; a loop that shares one copy of
// the transform's code took the same).
__global__ void __launch_bounds__(SEP_THREADS, 2) sep_desc_kernel(const __grid_constant__ SepTables tb,
                                                                  const SepItem* __restrict__ items, int nitem) {
    __shared__ SepBlock bk;
    __shared__ DF dsh[3 * SEP_THREADS / 32];
    if (!enter<true>(tb, items, nitem, bk, sep_smem, axis_x)) return;
    const SepLevel& lv = bk.lv;
    float2* sm = sep_smem;
    const int n = lv.n2, P2 = lv.P2;
    const int R = window_rows(lv);
    const int row0 = bk.block * lv.rowsW, rows = min(lv.rowsW, R - row0);
    const int pair = bk.a * lv.phases + bk.b;
    float2* V = lv.V + (int64_t)pair * lv.strideV + (int64_t)row0 * n;
    float2 dc = lv.dc[pair];
    for (int q = 1; q < lv.parts; ++q) {
        const DF d = df_add(DF{dc.x, dc.y}, DF{lv.dc[q].x, lv.dc[q].y});
        dc = make_float2(d.hi, d.lo);
    }
    // the window spectra, summed over sep_power's shares of the pairs
    auto spectrum = [&](int64_t e) {
        float2 v = V[e];
        for (int q = 1; q < lv.parts; ++q) v = caddf(v, V[e + q * lv.strideV]);
        return swapf(v);
    };
    const float scaleD = (float)lv.scaleD;
    float* desc = lv.desc + (int64_t)pair * lv.Khalf;
    // Kahan sums of this thread's residuals and targets
    float r2 = 0.f, r2c = 0.f, t2 = 0.f, t2c = 0.f;
    // writes the entry of (row l, rx) and returns the residual (0 outside the half window,
    // except at rx < 0 of row 0, the mirror of an entry of the same row)
    auto entry = [&](int l, int rx, float c) {
        int rz, ry;
        window_row(lv, row0 + l, rz, ry);
        int k = half_index(lv, rz, ry, rx);
        const bool mirror = k < 0 && rz == 0 && ry == 0;
        if (k < 0 && !(lv.fuse && mirror)) return 0.f;
        if (mirror) k = -rx;
        const float d = dc.x + fmaf(c, scaleD, dc.y);
        if (!mirror) desc[k] = d;
        if (lv.loss == nullptr) return 0.f;
        const float t = lv.sub[(int64_t)pair * lv.Khalf + k], rho = d - t;
        if (!mirror) {
            kahan_add(r2, r2c, rho * rho);
            kahan_add(t2, t2c, t * t);
        }
        return lv.scaleG * (k == 0 ? rho + rho : rho);
    };
    // embedded coefficient of position i of the row (both ends at the aliased rx = +-n/2)
    auto embedded = [&](int l, int i, float c) {
        float gsum = 0.f;
        if (i <= P2) gsum = entry(l, i, c);
        if (i > 0 && n - i <= P2) gsum += entry(l, i - n, c);
        return gsum;
    };
    // 3-D: row (0, -ry) holds the mirrored coefficients of (0, ry), i.e. the conjugate transform
    auto mirror_row = [&](int l) {
        int rz, ry;
        window_row(lv, row0 + l, rz, ry);
        return lv.n0 > 1 && rz == 0 && ry > 0 ? -2 * ry : 0;
    };
    auto skipped = [&](int l) {
        int rz, ry;
        window_row(lv, row0 + l, rz, ry);
        return rz == 0 && ry < 0;
    };
    if (lv.ax[2].fast) {
        for_pow2(lv.ax[2].fast, [&](auto cc) {
            constexpr int N = decltype(cc)::value, T = N / 8;
            constexpr bool WARP = T <= 32;
            const int line = threadIdx.x / T;
            const Line<N> ln = row_line<N>(sm, line, threadIdx.x % T, SEP_THREADS / T);
            const bool in = line < rows && !skipped(line);
            float2 v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = in ? spectrum(line * N + ln.t + e * T) : make_float2(0.f, 0.f);
            p2_fft<N, WARP, 0>(v, ln);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float gv = in ? embedded(line, ln.t + e * T, v[e].y) : 0.f;
                v[e] = make_float2(gv, 0.f);
            }
            if (!lv.fuse) return;
            if (p2_exchanges(N) & 1) line_sync<WARP>();
            p2_fft<N, WARP, 0>(v, ln);
            if (!in) return;
            const int m = mirror_row(line);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int i = ln.t + e * T;
                V[line * N + i] = v[e];
                if (m) V[(int64_t)(line + m) * N + i] = make_float2(v[e].x, -v[e].y);
            }
        });
    } else {
        const int pitch = spad(n - 1) + 2, wx = 2 * P2 + 1;
        const SepShared s = sep_shared(sm, n, lv.rowsW, pitch);
        const float inv_n = 1.0f / (float)n;
        for (int e = threadIdx.x; e < rows * n; e += blockDim.x) {
            const int l = fdiv(e, inv_n), i = e - l * n;
            s.a[l * pitch + spad(i)] = skipped(l) ? make_float2(0.f, 0.f) : spectrum(e);
        }
        float2* r = transform(lv.ax[2], s.a, s.b, s.tw, rows, pitch);
        if (!lv.fuse) {
            for (int e = threadIdx.x; e < rows * wx; e += blockDim.x) {
                const int l = e / wx, rx = e - l * wx - P2;
                entry(l, rx, r[l * pitch + spad(rx < 0 ? rx + n : rx)].y);
            }
        } else {
            for (int e = threadIdx.x; e < rows * n; e += blockDim.x) {
                const int l = fdiv(e, inv_n), i = e - l * n;
                float2& x = r[l * pitch + spad(i)];
                x = make_float2(skipped(l) ? 0.f : embedded(l, i, x.y), 0.f);
            }
            r = transform(lv.ax[2], r, r == s.a ? s.b : s.a, s.tw, rows, pitch);
            for (int e = threadIdx.x; e < rows * n; e += blockDim.x) {
                const int l = fdiv(e, inv_n), i = e - l * n;
                if (skipped(l)) continue;
                const float2 x = r[l * pitch + spad(i)];
                const int m = mirror_row(l);
                V[e] = x;
                if (m) V[(int64_t)(l + m) * n + i] = make_float2(x.x, -x.y);
            }
        }
    }
    if (lv.loss == nullptr) return;
    // Kahan's (sum, comp) stands for sum - comp
    DF sums[2] = {df_two_sum(r2, -r2c), df_two_sum(t2, -t2c)};
    block_sums_df(sums, dsh);
    const int blocks = (R + lv.rowsW - 1) / lv.rowsW;
    if (threadIdx.x == 0) lv.sums[lv.sumStart + pair * blocks + bk.block] = make_float4(sums[0].hi, sums[0].lo, sums[1].hi, sums[1].lo);
    loss_arrive(*lv.loss, lv.arrive, dsh);
}

// item: (level, phases a, b); blocks: groups of rowsW window rows.  G(r) of the row (the
// coefficient rule of the direct path's grid), embedded along x and transformed.
__global__ void __launch_bounds__(SEP_THREADS, 2) sep_gx_kernel(const __grid_constant__ SepTables tb,
                                                                const SepItem* __restrict__ items, int nitem) {
    __shared__ SepBlock bk;
    if (!enter<true>(tb, items, nitem, bk, sep_smem, axis_x)) return;
    const SepLevel& lv = bk.lv;
    float2* sm = sep_smem;
    const int n = lv.n2, P2 = lv.P2;
    const int R = window_rows(lv);
    const int row0 = bk.block * lv.rowsW, rows = min(lv.rowsW, R - row0);
    const int pair = bk.a * lv.phases + bk.b;
    const int64_t oab = (int64_t)pair * lv.Khalf, oba = ((int64_t)bk.b * lv.phases + bk.a) * lv.Khalf;
    const float scale = lv.scaleG * (lv.sc != nullptr ? lv.sc->gscale : 1.f);
    auto delta = [&](int64_t off, int k) {
        float d = lv.src[off + k] - (lv.sub != nullptr ? lv.sub[off + k] : 0.f);
        if (lv.tsum != nullptr) d = k == 0 ? d - lv.q / (1.f - lv.q) * *lv.tsum : d / (1.f - lv.q);
        return d;
    };
    auto G = [&](int rz, int ry, int rx) {
        const int k = half_index(lv, rz, ry, rx);
        if (k == 0) return scale * (delta(oab, 0) + delta(oba, 0));
        if (k > 0) return scale * delta(oab, k);
        return scale * delta(oba, half_index(lv, -rz, -ry, -rx));
    };
    auto embedded = [&](int l, int i) {
        int rz, ry;
        window_row(lv, row0 + l, rz, ry);
        float v = 0.f;
        if (i <= P2) v = G(rz, ry, i);
        if (i > 0 && n - i <= P2) v += G(rz, ry, i - n);
        return v;
    };
    float2* V = lv.V + (int64_t)pair * lv.strideV + (int64_t)row0 * n;
    if (lv.ax[2].fast) {
        for_pow2(lv.ax[2].fast, [&](auto cc) {
            constexpr int N = decltype(cc)::value, T = N / 8;
            constexpr bool WARP = T <= 32;
            const int line = threadIdx.x / T;
            const Line<N> ln = row_line<N>(sm, line, threadIdx.x % T, SEP_THREADS / T);
            const bool in = line < rows;
            float2 v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = make_float2(in ? embedded(line, ln.t + e * T) : 0.f, 0.f);
            p2_fft<N, WARP, 0>(v, ln);
            if (!in) return;
#pragma unroll
            for (int e = 0; e < 8; ++e) V[line * N + ln.t + e * T] = v[e];
        });
        return;
    }
    const int pitch = spad(n - 1) + 2;
    const SepShared s = sep_shared(sm, n, lv.rowsW, pitch);
    const float inv_n = 1.0f / (float)n;
    for (int e = threadIdx.x; e < rows * n; e += blockDim.x) {
        const int l = fdiv(e, inv_n), i = e - l * n;
        s.a[l * pitch + spad(i)] = make_float2(embedded(l, i), 0.f);
    }
    const float2* r = transform(lv.ax[2], s.a, s.b, s.tw, rows, pitch);
    for (int e = threadIdx.x; e < rows * n; e += blockDim.x) {
        const int l = fdiv(e, inv_n), i = e - l * n;
        V[e] = r[l * pitch + spad(i)];
    }
}

// ------------------------------------------------------------------------- last axis: products

namespace {

// Point i of G's column l of the phase pair (a, b), embedded along the last axis: rows
// r = 0 .. P of the pair, and at -r the conjugates of the pair (b, a) (G^ab(-r) = G^ba(r); both
// at r = +-n/2).
struct GCols {
    const float2 *ab, *ba;
    int P, n;
    int64_t stride;
    __device__ __forceinline__ GCols(const SepLevel& lv, int a, int b, const ColGroup& g) {
        P = lv.n0 > 1 ? lv.P0 : lv.P1;
        const float2* base = (lv.n0 > 1 ? lv.U : lv.V) + g.base;
        const int64_t size = lv.n0 > 1 ? lv.strideU : lv.strideV;
        ab = base + (a * lv.phases + b) * size;
        ba = base + (b * lv.phases + a) * size;
        n = g.n;
        stride = g.stride;
    }
    __device__ __forceinline__ float2 at(int i, int l) const {
        float2 v = make_float2(0.f, 0.f);
        if (i <= P) v = ab[i * stride + l];
        if (i > 0 && n - i <= P) {
            const float2 u = ba[(n - i) * stride + l];
            v = make_float2(v.x + u.x, v.y - u.y);
        }
        return v;
    }
};

}  // namespace

// item: (level, phase a).  Spectrum of G along the last axis, then for every feature pair the
// forward transform of the columns, the product sum_b conj(G^ab) Z^b and the inverse: Q^a, in
// place of Z for a single phase (G is even then: a real spectrum).  Its frequency 0, the sum of G over
// the window, is left for the term of F_u(M, c).  Bound by latency, as sep_power.
// 512^2, three levels, seven pairs: 23 us with the pairs shared among up to four blocks a group of
// columns, 29 without; 128^3, two levels: 100 us.
template <bool MULTI>
__global__ void __launch_bounds__(SEP_THREADS, MULTI ? 1 : 2)
sep_mul_kernel(const __grid_constant__ SepTables tb, const SepItem* __restrict__ items, int nitem) {
    __shared__ SepBlock bk;
    if (!enter<true>(tb, items, nitem, bk, sep_smem, axis_last)) return;
    const SepLevel& lv = bk.lv;
    float2* sm = sep_smem;
    const SepTier& t = tb.tier[bk.tier];
    if (bk.part * (last_ax(lv).fast ? SEP_BLOCK_PTS / (lv.colsL * last_ax(lv).n) : 1) >= t.npair) return;
    int x0, y;
    const ColGroup g = last_axis(lv, bk.block, x0, y);
    const SepAxis& ax = last_ax(lv);
    // of the unnormalised inverse; sep_desc's rows still lack the loss' factor
    const float gscale = lv.fuse && lv.sc != nullptr ? lv.sc->gscale : 1.f, norm = gscale / (float)lv.N;
    const bool has_sum = x0 == 0 && y == 0 && bk.part == 0 && threadIdx.x == 0;   // its first point is frequency 0
    if (ax.fast && (!MULTI || lv.phases <= SEP_FAST_PHASES)) {
        for_pow2(ax.fast, [&](auto cc) {
            constexpr int N = decltype(cc)::value, T = N / 8;
            constexpr int EX = p2_exchanges(N), PAR1 = EX & 1;
            const Cols<N> c(g.L);
            // MULTI: every phase's spectrum, this thread's points, behind the line buffers
            float2* gs = sep_smem + N + 2 * c.slots * c.L * sep_pitch(N, c.L) + threadIdx.x;
            float* gr = reinterpret_cast<float*>(sm + N + 2 * c.slots * c.L * sep_pitch(N, c.L)) + threadIdx.x;
            for (int b = 0; b < lv.phases; ++b) {
                const GCols gc(lv, bk.a, b, g);
                float2 v[8];
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    v[e] = c.l < g.cols ? gc.at(c.ln.t + e * T, c.l) : make_float2(0.f, 0.f);
                p2_fft<N, false, 0>(v, opaque(c.ln));
                if (PAR1) __syncthreads();
                if (has_sum) lv.gsum[bk.a * lv.phases + b] = gscale * v[0].x;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    if (MULTI) gs[(b * 8 + e) * SEP_THREADS] = make_float2(norm * v[e].x, -norm * v[e].y);
                    else gr[e * SEP_THREADS] = norm * v[e].x;
                }
            }
            for (int p0 = bk.part * c.slots; p0 < t.npair; p0 += bk.parts * c.slots) {
                const int p = p0 + c.slot;
                const bool on = p < t.npair;
                float2 v[8];
                if (!MULTI) {
                    load8<N>(lv.Z + (int64_t)p * lv.N, g, c, on, v);
                    if (!lv.keep) {              // else sep_power left the spectra
                        p2_fft<N, false, 0>(v, opaque(c.ln));
                        if (PAR1) __syncthreads();
                    }
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const float w = gr[e * SEP_THREADS];
                        v[e] = make_float2(w * v[e].y, w * v[e].x);
                    }
                    p2_fft<N, false, 0>(v, opaque(c.ln));
                    if (PAR1) __syncthreads();
                } else {
                    float2 acc[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) acc[e] = make_float2(0.f, 0.f);
                    for (int b = 0; b < lv.phases; ++b) {
                        load8<N>(lv.Z + ((int64_t)b * lv.maxPairs + p) * lv.N, g, c, on, v);
                        p2_fft<N, false, 0>(v, opaque(c.ln));
                        if (PAR1) __syncthreads();
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            const float2 w = gs[(b * 8 + e) * SEP_THREADS];
                            acc[e].x = fmaf(w.x, v[e].x, fmaf(-w.y, v[e].y, acc[e].x));
                            acc[e].y = fmaf(w.x, v[e].y, fmaf(w.y, v[e].x, acc[e].y));
                        }
                    }
#pragma unroll
                    for (int e = 0; e < 8; ++e) v[e] = swapf(acc[e]);
                    p2_fft<N, false, 0>(v, opaque(c.ln));
                    if (PAR1) __syncthreads();
                }
                swap8(v);
                store8<N>(lv.Q + ((int64_t)bk.a * lv.maxPairs + p) * lv.N, g, c, on, v);
            }
        });
        return;
    }
    const int pitch = sep_pitch(g.n, g.L), sh = 31 - __clz(g.L), total = g.L * g.n;
    const SepShared s = sep_shared(sm, g.n, g.L, pitch);
    float2* gs = s.b + g.L * pitch;              // the spectra of every b, own points
    auto own = [&](auto f) {
#pragma unroll
        for (int q = 0; q < SEP_OWN; ++q) {
            const int e = threadIdx.x + q * SEP_THREADS;
            if (e < total) f(q, e, (e & (g.L - 1)) * pitch + spad(e >> sh));
        }
    };
    for (int b = 0; b < lv.phases; ++b) {
        const GCols gc(lv, bk.a, b, g);
        __syncthreads();
        for (int e = threadIdx.x; e < total; e += blockDim.x) {
            const int l = e & (g.L - 1), i = e >> sh;
            s.a[l * pitch + spad(i)] = l < g.cols ? gc.at(i, l) : make_float2(0.f, 0.f);
        }
        const float2* r = transform(ax, s.a, s.b, s.tw, g.L, pitch);
        own([&](int, int e, int at) { gs[b * total + e] = make_float2(norm * r[at].x, MULTI ? -norm * r[at].y : 0.f); });
        if (has_sum) lv.gsum[bk.a * lv.phases + b] = gscale * r[0].x;
    }
    for (int p = bk.part; p < t.npair; p += bk.parts) {
        float2 acc[SEP_OWN];
#pragma unroll
        for (int q = 0; q < SEP_OWN; ++q) acc[q] = make_float2(0.f, 0.f);
        for (int b = 0; b < lv.phases; ++b) {
            __syncthreads();
            load_cols(lv.Z + ((int64_t)b * lv.maxPairs + p) * lv.N, g, pitch, s.a);
            const float2* r = s.a;
            if (MULTI || !lv.keep) r = transform(ax, s.a, s.b, s.tw, g.L, pitch);
            else __syncthreads();
            own([&](int q, int e, int at) {
                const float2 v = r[at], c = gs[b * total + e];
                acc[q].x = fmaf(c.x, v.x, fmaf(-c.y, v.y, acc[q].x));
                acc[q].y = fmaf(c.x, v.y, fmaf(c.y, v.x, acc[q].y));
            });
        }
        __syncthreads();
        own([&](int q, int, int at) { s.a[at] = swapf(acc[q]); });
        const float2* o = transform(ax, s.a, s.b, s.tw, g.L, pitch);
        float2* Q = lv.Q + ((int64_t)bk.a * lv.maxPairs + p) * lv.N;
        for (int e = threadIdx.x; e < total; e += blockDim.x) {
            const int l = e & (g.L - 1), i = e >> sh;
            if (l < g.cols) Q[g.base + i * g.stride + l] = swapf(o[l * pitch + spad(i)]);
        }
    }
}

// ------------------------------------------------------------------------- gradient

// item: (level, phase a); blocks: groups of rows.  Inverse along x of every feature pair and
// g(y) = F_u(M_y, c) sum G + sum_k s_k p_k'(M_y) Q_k(y), the slots' shares added in a fixed order.
// Bound by latency, as sep_feat.  Seven pairs: 512^2, three levels 28 us; 128^3, two levels 124 us,
// 5 of them for F_u(M, c) (coefficient gathers unrolled by three: 1 and 6 us more).
__global__ void __launch_bounds__(SEP_ROW_THREADS, 3) sep_grad_kernel(const __grid_constant__ SepTables tb,
                                                                      const SepItem* __restrict__ items, int nitem) {
    __shared__ SepBlock bk;
    if (!enter<true>(tb, items, nitem, bk, sep_smem, axis_x)) return;
    const SepLevel& lv = bk.lv;
    float2* sm = sep_smem;
    const SepTier& t = tb.tier[bk.tier];
    const float2* __restrict__ cf = tb.coef + t.coef;
    const int step = t.npair * t.nseg;
    const int rowsN = lv.n0 * lv.n1, n = lv.n2;
    const int row0 = bk.block * lv.rowsF, rows = min(lv.rowsF, rowsN - row0);
    const float* __restrict__ field = lv.field + (int64_t)bk.a * lv.N + (int64_t)row0 * n;
    const float2* __restrict__ Q = lv.Q + (int64_t)bk.a * lv.maxPairs * lv.N + (int64_t)row0 * n;
    float* __restrict__ part = lv.part + (int64_t)bk.a * lv.N + (int64_t)row0 * n;
    __shared__ float2 csh[MAX_PHASES];           // (c_b, sum_r G^ab(r))
    if (threadIdx.x < lv.phases) csh[threadIdx.x] = make_float2(lv.center[threadIdx.x], lv.gsum[bk.a * lv.phases + threadIdx.x]);
    // sum_b F_u(M, c_b) sum_r G^ab(r) at element o of the block's rows
    auto background = [&](int o) {
        const float M = field[o];
        float s = 0.f;
        for (int b = 0; b < lv.phases; ++b) {
            const float2 c = csh[b];
            float slope;
            pair_with(tb, M, c.x, slope);
            s = fmaf(slope, c.y, s);
        }
        return s;
    };
    __syncthreads();
    if (lv.ax[2].fast) {
        for_pow2(lv.ax[2].fast, [&](auto cc) {
            constexpr int N = decltype(cc)::value;
            using S = RowShape<N>;
            const int line = threadIdx.x / S::T, p = line % S::SLOTS, r0 = line / S::SLOTS;
            const Line<N> ln = row_line<N>(sm, line, threadIdx.x % S::T, S::LINES);
            float* red = reinterpret_cast<float*>(sm + N);      // over the line buffers: [slot][row][i]
            for (int rb = 0; rb < lv.rowsF; rb += S::ROWS) {
                const int row = rb + r0;
                const bool in = row < rows;
                float g[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) g[e] = 0.f;
                for (int p0 = 0; p0 < t.npair; p0 += S::SLOTS) {
                    const bool live = in && p0 + p < t.npair;
                    float2 v[8];
                    const float2* src = Q + (int64_t)(p0 + p) * lv.N + row * N + ln.t;
#pragma unroll
                    for (int e = 0; e < 8; ++e) v[e] = live ? swapf(src[e * S::T]) : make_float2(0.f, 0.f);
                    p2_fft<N, S::WARP, 0>(v, opaque(ln));
                    if (live) {
                        const float sg = p0 + p < t.npos ? (float)SEP_SEG : -(float)SEP_SEG;
                        // four positions at a time, located anew in every round: the state of eight
                        // does not fit the registers
#pragma unroll
                        for (int h = 0; h < 8; h += 4) {
                            float x[4], u[4];
                            int seg[4];
                            float2 f[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e) x[e] = field[row * N + ln.t + (h + e) * S::T];
                            locate<4>(t, x, seg, u);
                            eval_features<true, 4>(cf + (p0 + p) * t.nseg, step, t.nc, seg, u, f);
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                g[h + e] = fmaf(sg, fmaf(f[e].x, v[h + e].y, f[e].y * v[h + e].x), g[h + e]);
                        }
                    }
                    if (p2_exchanges(N) & 1) line_sync<S::WARP>();
                }
                if (S::SLOTS == 1) {
                    if (in) {
#pragma unroll
                        for (int e = 0; e < 8; ++e) part[row * N + ln.t + e * S::T] = g[e];
                        // (one at a time: eight side by side spill)
#pragma unroll 1
                        for (int e = 0; e < 8; ++e)
                            part[row * N + ln.t + e * S::T] += background(row * N + ln.t + e * S::T);
                    }
                    continue;
                }
                // the positions this thread finishes: their background terms before the barrier
                constexpr int FIN = (S::ROWS * N + SEP_ROW_THREADS - 1) / SEP_ROW_THREADS;
                const int here = min(S::ROWS, rows - rb) * N;
                float bg[FIN];
#pragma unroll
                for (int j = 0; j < FIN; ++j) {
                    const int o = threadIdx.x + j * SEP_ROW_THREADS;
                    bg[j] = o < here ? background(rb * N + o) : 0.f;
                }
                __syncthreads();
#pragma unroll
                for (int e = 0; e < 8; ++e) red[(p * S::ROWS + r0) * N + ln.t + e * S::T] = g[e];
                __syncthreads();
#pragma unroll
                for (int j = 0; j < FIN; ++j) {
                    const int o = threadIdx.x + j * SEP_ROW_THREADS;
                    if (o >= here) break;
                    float s = red[o];
#pragma unroll
                    for (int k = 1; k < S::SLOTS; ++k) s += red[k * S::ROWS * N + o];
                    part[rb * N + o] = s + bg[j];
                }
                __syncthreads();
            }
        });
        return;
    }
    const int pitch = spad(n - 1) + 2;
    const SepShared s = sep_shared(sm, n, lv.rowsF * SEP_SLOTS, pitch);
    const float inv_n = 1.0f / (float)n;
    float g[SEP_OWN];
#pragma unroll
    for (int q = 0; q < SEP_OWN; ++q) g[q] = 0.f;
    for (int p0 = 0; p0 < t.npair; p0 += SEP_SLOTS) {
        const int nc = min(SEP_SLOTS, t.npair - p0);
        __syncthreads();
        for (int e = threadIdx.x; e < rows * nc * n; e += blockDim.x) {
            const int q = fdiv(e, inv_n), i = e - q * n;
            const int l = q / nc, c = q - l * nc;
            s.a[q * pitch + spad(i)] = swapf(Q[(int64_t)(p0 + c) * lv.N + l * n + i]);
        }
        const float2* r = transform(lv.ax[2], s.a, s.b, s.tw, rows * nc, pitch);
#pragma unroll
        for (int q = 0; q < SEP_OWN; ++q) {
            const int e = threadIdx.x + q * SEP_ROW_THREADS;
            if (e < rows * n) {
                const int l = fdiv(e, inv_n), i = e - l * n;
                const float x[1] = {field[e]};
                float u[1];
                int seg[1];
                locate<1>(t, x, seg, u);
                for (int c = 0; c < nc; ++c) {
                    float2 f[1];
                    eval_features<true, 1>(cf + (p0 + c) * t.nseg, step, t.nc, seg, u, f);
                    const float2 v = r[(l * nc + c) * pitch + spad(i)];
                    g[q] = fmaf(p0 + c < t.npos ? (float)SEP_SEG : -(float)SEP_SEG, fmaf(f[0].x, v.y, f[0].y * v.x), g[q]);
                }
            }
        }
    }
#pragma unroll
    for (int q = 0; q < SEP_OWN; ++q) {
        const int e = threadIdx.x + q * SEP_ROW_THREADS;
        if (e < rows * n) part[e] = g[q] + background(e);
    }
}

// ------------------------------------------------------------------------- launchers

namespace {
size_t bytes_of(int n, int lines, int pitch) { return (size_t)(((n + 1) & ~1) + 2 * lines * pitch) * sizeof(float2); }
// power-of-two rows: the block's whole line capacity (row_pitch)
size_t fast_row_bytes(int n, int threads) {
    int p = n - 1 + (n - 1) / 16 + 1;
    const int want = n >= 128 ? 0 : n / 8;
    while (p % 16 != want) ++p;
    return bytes_of(n, 8 * threads / n, p);
}
}  // namespace

size_t sep_smem_feat(const SepLevel& lv) {
    const int n = lv.n2;
    return lv.ax[2].fast ? fast_row_bytes(n, SEP_ROW_THREADS)
                         : bytes_of(n, lv.rowsF * SEP_SLOTS, n - 1 + ((n - 1) >> 4) + 2);
}
size_t sep_smem_window(const SepLevel& lv) {
    const int n = lv.n2;
    return lv.ax[2].fast ? fast_row_bytes(n, SEP_THREADS) : bytes_of(n, lv.rowsW, n - 1 + ((n - 1) >> 4) + 2);
}
size_t sep_smem_y(const SepLevel& lv) {
    const int lines = lv.ax[1].fast ? SEP_BLOCK_PTS / lv.n1 : lv.colsY;
    return bytes_of(lv.n1, lines, sep_pitch(lv.n1, lv.colsY));
}
size_t sep_smem_last(const SepLevel& lv, bool mul) {
    const SepAxis& ax = lv.n0 > 1 ? lv.ax[0] : lv.ax[1];
    const int lines = ax.fast ? SEP_BLOCK_PTS / ax.n : lv.colsL;
    size_t b = bytes_of(ax.n, lines, sep_pitch(ax.n, lv.colsL));
    if (ax.fast && lv.phases == 1) b += (size_t)SEP_BLOCK_PTS * sizeof(float);      // a thread's own eight values
    if (mul) {
        if (!ax.fast || lv.phases > SEP_FAST_PHASES) b = bytes_of(ax.n, lv.colsL, sep_pitch(ax.n, lv.colsL)) +
                                                         (size_t)lv.phases * lv.colsL * ax.n * sizeof(float2);
        else if (lv.phases > 1) b += (size_t)lv.phases * SEP_BLOCK_PTS * sizeof(float2);
    }
    return b;
}

void launch_sep(SepKernel k, const SepTables& tb, const SepItem* items, int nitem, int64_t blocks, size_t smem,
                cudaStream_t s) {
    if (blocks <= 0) return;
    const unsigned b = (unsigned)blocks;
    constexpr int T = SEP_THREADS;
    switch (k) {
        case SEP_FEAT: launch_dep(sep_feat_kernel, b, SEP_ROW_THREADS, smem, s, tb, items, nitem); break;
        case SEP_FFT_Y: launch_dep(sep_fft_y_kernel<false>, b, T, smem, s, tb, items, nitem); break;
        case SEP_POWER: launch_dep(sep_power_kernel<false>, b, T, smem, s, tb, items, nitem); break;
        case SEP_POWER_PH: launch_dep(sep_power_kernel<true>, b, T, smem, s, tb, items, nitem); break;
        case SEP_INV_Y: launch_dep(sep_win_y_kernel<true>, b, T, smem, s, tb, items, nitem); break;
        case SEP_DESC: launch_dep(sep_desc_kernel, b, T, smem, s, tb, items, nitem); break;
        case SEP_GX: launch_dep(sep_gx_kernel, b, T, smem, s, tb, items, nitem); break;
        case SEP_GY: launch_dep(sep_win_y_kernel<false>, b, T, smem, s, tb, items, nitem); break;
        case SEP_MUL: launch_dep(sep_mul_kernel<false>, b, T, smem, s, tb, items, nitem); break;
        case SEP_MUL_PH: launch_dep(sep_mul_kernel<true>, b, T, smem, s, tb, items, nitem); break;
        case SEP_IFFT_Y: launch_dep(sep_fft_y_kernel<true>, b, T, smem, s, tb, items, nitem); break;
        case SEP_GRAD: launch_dep(sep_grad_kernel, b, SEP_ROW_THREADS, smem, s, tb, items, nitem); break;
        default: break;
    }
}

void set_sep_attributes() {
    const void* ks[] = {(const void*)sep_feat_kernel,         (const void*)sep_fft_y_kernel<false>,
                        (const void*)sep_fft_y_kernel<true>,  (const void*)sep_power_kernel<false>,
                        (const void*)sep_power_kernel<true>,  (const void*)sep_win_y_kernel<true>,
                        (const void*)sep_win_y_kernel<false>, (const void*)sep_desc_kernel,
                        (const void*)sep_gx_kernel,           (const void*)sep_mul_kernel<false>,
                        (const void*)sep_mul_kernel<true>,    (const void*)sep_grad_kernel};
    for (const void* k : ks) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SEP_MAX_SMEM);
}

}  // namespace dmcr
