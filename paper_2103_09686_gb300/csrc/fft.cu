// FFT path of the descriptor (sm_103a): the periodic autocorrelation
//     C(r) = (1/N) sum_x M_x M_{x+r} = (1/N) IDFT( |DFT(M)|^2 )(r)
// gives, exactly up to rounding,
//   * the identity-threshold descriptor (f(x) = x, the ablation of Sec. 4.1):
//         S_bar(r) = ( <M^2> + C(r) ) / 2,   <M^2> = C(0);
//   * the soft-threshold descriptor of a BINARY field (App. A):
//         S_bar(r) = (1 - 2 f(1/2)^2) C(r) + 2 f(1/2)^2 C(0)  (r != 0),   S_bar(0) = C(0),
//     used to characterise binary targets;
// and the identity-threshold adjoint as one cross-correlation,
//         g(y) = ( M_y sum_r A(r) + sum_r A(r) M_{y+r} ) / 2,
//         sum_r A(r) M_{y+r} = (1/N) IDFT( DFT(M) DFT(A) )(y)       (A even: DFT(A) real).
// Hand-written mixed-radix (8, 4, 2, 3, 5) Stockham transforms in FP64 (the descriptor needs
// ~1e-7 relative accuracy on C(r)).
//
// The path is bound by the FP64 pipe (1.7 operations per SM and clock), so it computes only what
// is used: the field and A are real, so two rows share one complex transform along x and only the
// n2/2 + 1 columns of the half spectrum go on; the correlation is needed on the window alone, so
// after the inverse along the last axis (z in 3-D, y in 2-D) only r = 0 .. P planes are kept, and
// A's transform starts from the same few rows; the power spectrum and the product are formed
// where the last axis is transformed, without a pass of their own.
//   fft_rows    rows of M in pairs -> X[z][y][kx]; sum M^2
//   fft_y       3-D: transform along y, in place
//   fft_last    last axis: transform (X stays), |X|^2, inverse, cropped
//   fft_win_y   3-D: inverse along y cropped to the window / A's rows embedded and transformed
//   fft_desc    inverse along x, two window rows at a time: the descriptor
//   fft_coef    rows of A in pairs along x
//   fft_mul     last axis: transform of A, product with X, inverse
//   fft_grad    inverse along x, two rows at a time: the gradient
// 128^3, +-24, loss and gradient: 1715 us with twelve full complex passes of 130 us and seven
// elementwise kernels, 579 us so.
#include <algorithm>

#include "common.cuh"

namespace dmcr {

namespace {

constexpr int FFT_THREADS = 256;

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(fma(a.x, b.x, -(a.y * b.y)), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cswap(double2 a) { return make_double2(a.y, a.x); }
__device__ __forceinline__ double2 conj2(double2 a) { return make_double2(a.x, -a.y); }
// multiply by -i
__device__ __forceinline__ double2 mul_mi(double2 a) { return make_double2(a.y, -a.x); }

__device__ __forceinline__ void bfly4(double2& a, double2& b, double2& c, double2& d) {
    const double2 s0 = cadd(a, c), d0 = csub(a, c), s1 = cadd(b, d), d1 = mul_mi(csub(b, d));
    a = cadd(s0, s1);
    b = cadd(d0, d1);
    c = csub(s0, s1);
    d = csub(d0, d1);
}

// One forward Stockham stage of radix R over `lines` lines of n points in shared memory
// (src -> dst): every butterfly reads R values n/R apart, multiplies by the twiddles of its
// offset k within the current sub-transform length Ns, and writes R values Ns apart.
template <int R>
__device__ __forceinline__ void fft_stage(const FftAxis& ax, const double2* __restrict__ src,
                                          double2* __restrict__ dst, int lines, int Ns) {
    const int n = ax.n, nR = n / R, tstep = nR / Ns;
    for (int t = threadIdx.x; t < lines * nR; t += FFT_THREADS) {
        const int l = t / nR, j = t - l * nR;
        const int k = j % Ns;
        const double2* in = src + l * n;
        double2 v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = in[j + r * nR];
        if (Ns > 1) {
#pragma unroll
            for (int r = 1; r < R; ++r) v[r] = cmul(v[r], ax.tw[k * r * tstep]);
        }
        double2 V[R];
        if constexpr (R == 2) {
            V[0] = cadd(v[0], v[1]);
            V[1] = csub(v[0], v[1]);
        } else if constexpr (R == 4) {
            bfly4(v[0], v[1], v[2], v[3]);
#pragma unroll
            for (int q = 0; q < 4; ++q) V[q] = v[q];
        } else if constexpr (R == 8) {
            bfly4(v[0], v[2], v[4], v[6]);
            bfly4(v[1], v[3], v[5], v[7]);
            constexpr double h = 0.70710678118654752440;
            const double2 w1 = make_double2(v[3].x + v[3].y, v[3].y - v[3].x);     // odd 1 times (1 - i)
            const double2 w2 = mul_mi(v[5]);
            const double2 w3 = make_double2(v[7].y - v[7].x, -v[7].x - v[7].y);    // odd 3 times -(1 + i)
            V[0] = cadd(v[0], v[1]);
            V[4] = csub(v[0], v[1]);
            V[1] = make_double2(fma(h, w1.x, v[2].x), fma(h, w1.y, v[2].y));
            V[5] = make_double2(fma(-h, w1.x, v[2].x), fma(-h, w1.y, v[2].y));
            V[2] = cadd(v[4], w2);
            V[6] = csub(v[4], w2);
            V[3] = make_double2(fma(h, w3.x, v[6].x), fma(h, w3.y, v[6].y));
            V[7] = make_double2(fma(-h, w3.x, v[6].x), fma(-h, w3.y, v[6].y));
        } else {
            // radix 3 and 5: V[q] = sum_r v[r] exp(-2 pi i r q / R), r paired with R - r
            constexpr double c3 = -0.5, s3 = 0.86602540378443864676;
            constexpr double c51 = 0.30901699437494742410, c52 = -0.80901699437494742410,
                             s51 = 0.95105651629515357212, s52 = 0.58778525229247312917;
            if constexpr (R == 3) {
                const double2 p = cadd(v[1], v[2]), m = mul_mi(csub(v[1], v[2]));
                const double2 a = make_double2(fma(c3, p.x, v[0].x), fma(c3, p.y, v[0].y));
                V[0] = cadd(v[0], p);
                V[1] = make_double2(fma(s3, m.x, a.x), fma(s3, m.y, a.y));
                V[2] = make_double2(fma(-s3, m.x, a.x), fma(-s3, m.y, a.y));
            } else {
                const double2 p1 = cadd(v[1], v[4]), m1 = mul_mi(csub(v[1], v[4]));
                const double2 p2 = cadd(v[2], v[3]), m2 = mul_mi(csub(v[2], v[3]));
                V[0] = cadd(v[0], cadd(p1, p2));
                const double2 a1 = make_double2(fma(c51, p1.x, fma(c52, p2.x, v[0].x)), fma(c51, p1.y, fma(c52, p2.y, v[0].y)));
                const double2 a2 = make_double2(fma(c52, p1.x, fma(c51, p2.x, v[0].x)), fma(c52, p1.y, fma(c51, p2.y, v[0].y)));
                const double2 b1 = make_double2(fma(s51, m1.x, s52 * m2.x), fma(s51, m1.y, s52 * m2.y));
                const double2 b2 = make_double2(fma(s52, m1.x, -(s51 * m2.x)), fma(s52, m1.y, -(s51 * m2.y)));
                V[1] = cadd(a1, b1);
                V[4] = csub(a1, b1);
                V[2] = cadd(a2, b2);
                V[3] = csub(a2, b2);
            }
        }
        double2* out = dst + l * n + (j - k) * R + k;
#pragma unroll
        for (int q = 0; q < R; ++q) out[q * Ns] = V[q];
    }
}

// Forward transform of `lines` lines from `a`, through `b` and back; returns the buffer that holds
// the result.  Begins and ends with a barrier.  An inverse exchanges real and imaginary parts
// of its input and output.
__device__ __noinline__ double2* fft_lines(const FftAxis& ax, double2* a, double2* b, int lines) {
    int Ns = 1;
    __syncthreads();
    for (int s = 0; s < ax.nrad; ++s) {
        const int R = ax.rad[s];
        switch (R) {
            case 8: fft_stage<8>(ax, a, b, lines, Ns); break;
            case 4: fft_stage<4>(ax, a, b, lines, Ns); break;
            case 2: fft_stage<2>(ax, a, b, lines, Ns); break;
            case 3: fft_stage<3>(ax, a, b, lines, Ns); break;
            default: fft_stage<5>(ax, a, b, lines, Ns); break;
        }
        Ns *= R;
        double2* x = a;
        a = b;
        b = x;
        __syncthreads();
    }
    return a;
}

extern __shared__ __align__(16) double2 fft_smem[];

// Canonical half-window index of (rz, ry, rx), -1 if it is not in the half window.
__device__ __forceinline__ int64_t fft_half_index(const FftArgs& g, int rz, int ry, int rx) {
    const int Px = g.P2, Py = g.P1;
    if (rz == 0 && ry == 0) return rx >= 0 ? rx : -1;
    if (rz == 0) return ry > 0 ? (Px + 1) + (int64_t)(ry - 1) * (2 * Px + 1) + (rx + Px) : -1;
    if (rz < 0) return -1;
    return (Px + 1) + (int64_t)Py * (2 * Px + 1) + ((int64_t)(rz - 1) * (2 * Py + 1) + (ry + Py)) * (2 * Px + 1) +
           (rx + Px);
}

// rows kept of the window -> (rz, ry): 3-D rz = 0 .. P0 and every ry, 2-D ry = 0 .. P1
__device__ __forceinline__ void fft_window_row(const FftArgs& g, int row, int& rz, int& ry) {
    if (g.n0 > 1) {
        const int wy = 2 * g.P1 + 1;
        rz = row / wy;
        ry = row - rz * wy - g.P1;
    } else {
        rz = 0;
        ry = row;
    }
}
__device__ __forceinline__ int fft_window_rows(const FftArgs& g) {
    return g.n0 > 1 ? (g.P0 + 1) * (2 * g.P1 + 1) : g.P1 + 1;
}

// fixed-order sum over the block (FFT_THREADS threads); valid in every thread
__device__ __forceinline__ double block_sum(double v, double* sh) {
    __syncthreads();
    sh[threadIdx.x] = v;
    for (int w = FFT_THREADS / 2; w > 0; w >>= 1) {
        __syncthreads();
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    }
    __syncthreads();
    return sh[0];
}

// Half spectra of two real lines from the transform Z of (first + i second).
__device__ __forceinline__ void unpack(const double2* r, int n, int k, double2& A, double2& B) {
    const double2 z = r[k], y = r[k == 0 ? 0 : n - k];
    A = make_double2(0.5 * (z.x + y.x), 0.5 * (z.y - y.y));
    B = make_double2(0.5 * (z.y + y.y), 0.5 * (y.x - z.x));
}
// The transform of (first + i second) at k from their half spectra, exchanged for an inverse.
__device__ __forceinline__ double2 pack_swapped(const double2* A, const double2* B, int n, int nh, int k) {
    double2 a, b;
    if (k < nh) {
        a = A[k];
        b = B != nullptr ? B[k] : make_double2(0.0, 0.0);
    } else {
        a = conj2(A[n - k]);
        b = B != nullptr ? conj2(B[n - k]) : make_double2(0.0, 0.0);
    }
    return make_double2(a.y + b.x, a.x - b.y);       // swapped (a.x - b.y, a.y + b.x)
}

}  // namespace

// tw[t] = exp(-2 pi i t / len) of the three axes, one block column per axis
__global__ void fft_twiddle_kernel(FftArgs g) {
    dep_wait();
    dep_trigger();
    const FftAxis& ax = g.ax[blockIdx.y];
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ax.n) return;
    double sv, cv;
    sincospi(2.0 * (double)t / (double)ax.n, &sv, &cv);
    ax.tw[t] = make_double2(cv, -sv);
}

// Row pairs of the field along x; the block's share of sum M^2.
__global__ void __launch_bounds__(FFT_THREADS, 3) fft_rows_kernel(const __grid_constant__ FftArgs g) {
    dep_wait();
    dep_trigger();
    __shared__ double sh[FFT_THREADS];
    const int n = g.n2, nh = g.nh, L = g.Lx;
    const int64_t rows = (int64_t)g.n0 * g.n1, q0 = (int64_t)blockIdx.x * L;
    const int lines = (int)min((int64_t)L, (rows + 1) / 2 - q0);
    double2 *a = fft_smem, *b = fft_smem + L * n;
    double sq = 0.0;
    for (int e = threadIdx.x; e < lines * n; e += FFT_THREADS) {
        const int l = e / n, i = e - l * n;
        const int64_t row = 2 * (q0 + l);
        const float u = g.field[row * n + i], v = row + 1 < rows ? g.field[(row + 1) * n + i] : 0.f;
        a[e] = make_double2((double)u, (double)v);
        sq = fma((double)u, (double)u, fma((double)v, (double)v, sq));
    }
    const double2* r = fft_lines(g.ax[2], a, b, lines);
    for (int e = threadIdx.x; e < lines * nh; e += FFT_THREADS) {
        const int l = e / nh, k = e - l * nh;
        const int64_t row = 2 * (q0 + l);
        double2 A, B;
        unpack(r + l * n, n, k, A, B);
        g.X[row * nh + k] = A;
        if (row + 1 < rows) g.X[(row + 1) * nh + k] = B;
    }
    sq = block_sum(sq, sh);
    if (threadIdx.x == 0) g.sq[blockIdx.x] = sq;
}

// columns of one block along a strided axis: L adjacent kx
struct FftCols {
    int n, L, cols;
    int64_t base, stride;
};

__device__ __forceinline__ void fft_load(const double2* __restrict__ src, const FftCols& c, bool swap, double2* a) {
    for (int e = threadIdx.x; e < c.L * c.n; e += FFT_THREADS) {
        const int i = e / c.L, l = e - i * c.L;
        const double2 v = l < c.cols ? src[c.base + i * c.stride + l] : make_double2(0.0, 0.0);
        a[l * c.n + i] = swap ? cswap(v) : v;
    }
}

// Middle axis of 3-D, in place.
template <bool INVERSE>
__global__ void __launch_bounds__(FFT_THREADS, 3) fft_y_kernel(const __grid_constant__ FftArgs g) {
    dep_wait();
    dep_trigger();
    const int xg = (g.nh + g.Ly - 1) / g.Ly, x0 = (int)(blockIdx.x % xg) * g.Ly, z = (int)(blockIdx.x / xg);
    const FftCols c{g.n1, g.Ly, min(g.Ly, g.nh - x0), (int64_t)z * g.n1 * g.nh + x0, g.nh};
    double2 *a = fft_smem, *b = fft_smem + c.L * c.n;
    fft_load(g.X, c, INVERSE, a);
    const double2* r = fft_lines(g.ax[1], a, b, c.L);
    for (int e = threadIdx.x; e < c.L * c.n; e += FFT_THREADS) {
        const int i = e / c.L, l = e - i * c.L;
        if (l < c.cols) g.X[c.base + i * c.stride + l] = INVERSE ? cswap(r[l * c.n + i]) : r[l * c.n + i];
    }
}

__device__ __forceinline__ FftCols fft_last_cols(const FftArgs& g) {
    const int xg = (g.nh + g.Ll - 1) / g.Ll, x0 = (int)(blockIdx.x % xg) * g.Ll, y = (int)(blockIdx.x / xg);
    const bool d3 = g.n0 > 1;
    return FftCols{d3 ? g.n0 : g.n1, g.Ll, min(g.Ll, g.nh - x0), (int64_t)y * g.nh + x0,
                   d3 ? (int64_t)g.n1 * g.nh : (int64_t)g.nh};
}

// Last axis: X's transform (left in place), the power spectrum and its inverse, rows 0 .. P.
__global__ void __launch_bounds__(FFT_THREADS, 3) fft_last_kernel(const __grid_constant__ FftArgs g) {
    dep_wait();
    dep_trigger();
    const FftCols c = fft_last_cols(g);
    const FftAxis& ax = g.n0 > 1 ? g.ax[0] : g.ax[1];
    double2 *a = fft_smem, *b = fft_smem + c.L * c.n;
    fft_load(g.X, c, false, a);
    double2* r = fft_lines(ax, a, b, c.L);
    for (int e = threadIdx.x; e < c.L * c.n; e += FFT_THREADS) {
        const int i = e / c.L, l = e - i * c.L;
        const double2 v = r[l * c.n + i];
        if (l < c.cols) g.X[c.base + i * c.stride + l] = v;
        r[l * c.n + i] = make_double2(0.0, fma(v.x, v.x, v.y * v.y));      // exchanged
    }
    const double2* o = fft_lines(ax, r, r == a ? b : a, c.L);
    const int P = g.n0 > 1 ? g.P0 : g.P1;
    double2* out = g.n0 > 1 ? g.U : g.V;
    for (int e = threadIdx.x; e < c.L * (P + 1); e += FFT_THREADS) {
        const int i = e / c.L, l = e - i * c.L;
        if (l < c.cols) out[c.base + i * c.stride + l] = cswap(o[l * c.n + i]);
    }
}

// 3-D: middle axis of the window.  DESC: U -> V, inverse cropped to -P1 .. P1.  Otherwise V -> U:
// A's rows embedded (both ends at the aliased +-n/2) and transformed.
template <bool DESC>
__global__ void __launch_bounds__(FFT_THREADS, 3) fft_win_y_kernel(const __grid_constant__ FftArgs g) {
    dep_wait();
    dep_trigger();
    const int xg = (g.nh + g.Lw - 1) / g.Lw, x0 = (int)(blockIdx.x % xg) * g.Lw, rz = (int)(blockIdx.x / xg);
    const int n = g.n1, L = g.Lw, cols = min(L, g.nh - x0), wy = 2 * g.P1 + 1;
    double2 *a = fft_smem, *b = fft_smem + L * n;
    double2* U = g.U + (int64_t)rz * g.n1 * g.nh + x0;
    double2* V = g.V + (int64_t)rz * wy * g.nh + x0;
    for (int e = threadIdx.x; e < L * n; e += FFT_THREADS) {
        const int i = e / L, l = e - i * L;
        double2 v = make_double2(0.0, 0.0);
        if (l < cols) {
            if (DESC) {
                v = cswap(U[(int64_t)i * g.nh + l]);
            } else {
                if (i <= g.P1) v = V[(int64_t)(i + g.P1) * g.nh + l];
                if (i > 0 && n - i <= g.P1) v = cadd(v, V[(int64_t)(i - n + g.P1) * g.nh + l]);
            }
        }
        a[l * n + i] = v;
    }
    const double2* r = fft_lines(g.ax[1], a, b, L);
    for (int e = threadIdx.x; e < L * (DESC ? wy : n); e += FFT_THREADS) {
        const int i = e / L, l = e - i * L;
        if (l >= cols) continue;
        if (DESC) {
            const int ry = i - g.P1;
            V[(int64_t)i * g.nh + l] = cswap(r[l * n + (ry < 0 ? ry + n : ry)]);
        } else {
            U[(int64_t)i * g.nh + l] = r[l * n + i];
        }
    }
}

// Pairs of window rows, inverse along x: desc[k] = w S_bar(r_k) (mode 0: identity threshold;
// mode 1: soft threshold of a binary field, App. A with fh2 = f(1/2)^2).
__global__ void __launch_bounds__(FFT_THREADS, 3) fft_desc_kernel(const __grid_constant__ FftArgs g) {
    dep_wait();
    dep_trigger();
    __shared__ double sh[FFT_THREADS];
    const int n = g.n2, nh = g.nh, L = g.Lv, R = fft_window_rows(g), q0 = blockIdx.x * L;
    const int lines = min(L, (R + 1) / 2 - q0);
    double2 *a = fft_smem, *b = fft_smem + L * n;
    double s = 0.0;
    for (int i = threadIdx.x; i < g.nsq; i += FFT_THREADS) s += g.sq[i];
    const double C0 = block_sum(s, sh) / (double)g.N;
    for (int e = threadIdx.x; e < lines * n; e += FFT_THREADS) {
        const int l = e / n, k = e - l * n, row = 2 * (q0 + l);
        const double2* A = g.V + (int64_t)row * nh;
        a[e] = pack_swapped(A, row + 1 < R ? A + nh : nullptr, n, nh, k);
    }
    const double2* r = fft_lines(g.ax[2], a, b, lines);
    const double invN2 = 1.0 / ((double)g.N * (double)g.N);
    const int wx = 2 * g.P2 + 1;
    for (int e = threadIdx.x; e < 2 * lines * wx; e += FFT_THREADS) {
        const int h = e / wx, rx = e - h * wx - g.P2, row = 2 * q0 + h;
        if (row >= R) continue;
        int rz, ry;
        fft_window_row(g, row, rz, ry);
        const int64_t k = fft_half_index(g, rz, ry, rx);
        if (k < 0) continue;
        const double2 v = r[(h / 2) * n + (rx < 0 ? rx + n : rx)];
        const double Cr = (h & 1 ? v.x : v.y) * invN2;       // exchanged: the first row is the imaginary part
        double S;
        if (g.mode == 0) S = k == 0 ? C0 : 0.5 * (C0 + Cr);
        else S = k == 0 ? C0 : (1.0 - 2.0 * g.fh2) * Cr + 2.0 * g.fh2 * C0;
        g.desc[k] = (float)((double)g.weight * S);
    }
}

// Pairs of window rows of A (plane 0 of the dense coefficient grid) embedded along x.
__global__ void __launch_bounds__(FFT_THREADS, 3) fft_coef_kernel(const __grid_constant__ FftArgs g) {
    dep_wait();
    dep_trigger();
    const int n = g.n2, nh = g.nh, L = g.Lv, R = fft_window_rows(g), q0 = blockIdx.x * L;
    const int lines = min(L, (R + 1) / 2 - q0);
    double2 *a = fft_smem, *b = fft_smem + L * n;
    auto A = [&](int row, int i) {
        if (row >= R) return 0.0;
        int rz, ry;
        fft_window_row(g, row, rz, ry);
        const float* p = g.Gd + ((int64_t)(rz + g.P0) * (2 * g.P1 + 1) + (ry + g.P1)) * g.NB * GBLOCK;
        double v = 0.0;
        if (i <= g.P2) v = (double)p[((i + g.P2) / T) * GBLOCK + 4 * ((i + g.P2) % T)];
        if (i > 0 && n - i <= g.P2) v += (double)p[((i - n + g.P2) / T) * GBLOCK + 4 * ((i - n + g.P2) % T)];
        return v;
    };
    for (int e = threadIdx.x; e < lines * n; e += FFT_THREADS) {
        const int l = e / n, i = e - l * n, row = 2 * (q0 + l);
        a[e] = make_double2(A(row, i), A(row + 1, i));
    }
    const double2* r = fft_lines(g.ax[2], a, b, lines);
    for (int e = threadIdx.x; e < lines * nh; e += FFT_THREADS) {
        const int l = e / nh, k = e - l * nh, row = 2 * (q0 + l);
        double2 u, v;
        unpack(r + l * n, n, k, u, v);
        g.V[(int64_t)row * nh + k] = u;
        if (row + 1 < R) g.V[(int64_t)(row + 1) * nh + k] = v;
    }
}

// Last axis: transform of A (real, since A is even: row -r is the conjugate of row r), product
// with X (transformed here first when no descriptor of the same call left it so), inverse, in
// place; sum_r A(r) = DFT(A)(0).
__global__ void __launch_bounds__(FFT_THREADS, 3) fft_mul_kernel(const __grid_constant__ FftArgs g) {
    dep_wait();
    dep_trigger();
    const FftCols c = fft_last_cols(g);
    const FftAxis& ax = g.n0 > 1 ? g.ax[0] : g.ax[1];
    const int P = g.n0 > 1 ? g.P0 : g.P1;
    const double2* src = g.n0 > 1 ? g.U : g.V;
    double2 *a = fft_smem, *b = fft_smem + c.L * c.n;
    double* w = reinterpret_cast<double*>(b + c.L * c.n);
    for (int e = threadIdx.x; e < c.L * c.n; e += FFT_THREADS) {
        const int i = e / c.L, l = e - i * c.L;
        double2 v = make_double2(0.0, 0.0);
        if (l < c.cols) {
            if (i <= P) v = src[c.base + i * c.stride + l];
            if (i > 0 && c.n - i <= P) v = cadd(v, conj2(src[c.base + (c.n - i) * c.stride + l]));
        }
        a[l * c.n + i] = v;
    }
    double2* r = fft_lines(ax, a, b, c.L);
    for (int e = threadIdx.x; e < c.L * c.n; e += FFT_THREADS) w[e] = r[e].x;
    if (blockIdx.x == 0 && threadIdx.x == 0) *g.dc = r[0].x;
    __syncthreads();
    fft_load(g.X, c, false, a);
    r = a;
    if (!g.x_ready) r = fft_lines(ax, a, b, c.L);
    else __syncthreads();
    for (int e = threadIdx.x; e < c.L * c.n; e += FFT_THREADS) {
        const double2 v = r[e];
        r[e] = make_double2(w[e] * v.y, w[e] * v.x);         // exchanged
    }
    const double2* o = fft_lines(ax, r, r == a ? b : a, c.L);
    for (int e = threadIdx.x; e < c.L * c.n; e += FFT_THREADS) {
        const int i = e / c.L, l = e - i * c.L;
        if (l < c.cols) g.X[c.base + i * c.stride + l] = cswap(o[l * c.n + i]);
    }
}

// Row pairs, inverse along x: part[y] = ( M_y sum_r A(r) + Z[y] / N ) / 2.
__global__ void __launch_bounds__(FFT_THREADS, 3) fft_grad_kernel(const __grid_constant__ FftArgs g) {
    dep_wait();
    dep_trigger();
    const int n = g.n2, nh = g.nh, L = g.Lx;
    const int64_t rows = (int64_t)g.n0 * g.n1, q0 = (int64_t)blockIdx.x * L;
    const int lines = (int)min((int64_t)L, (rows + 1) / 2 - q0);
    double2 *a = fft_smem, *b = fft_smem + L * n;
    for (int e = threadIdx.x; e < lines * n; e += FFT_THREADS) {
        const int l = e / n, k = e - l * n;
        const int64_t row = 2 * (q0 + l);
        const double2* A = g.X + row * nh;
        a[e] = pack_swapped(A, row + 1 < rows ? A + nh : nullptr, n, nh, k);
    }
    const double2* r = fft_lines(g.ax[2], a, b, lines);
    const double half_sum = 0.5 * *g.dc, scale = 0.5 / (double)g.N;
    for (int e = threadIdx.x; e < lines * n; e += FFT_THREADS) {
        const int l = e / n, i = e - l * n;
        const int64_t row = 2 * (q0 + l), y = row * n + i;
        g.part[y] = (float)fma((double)g.field[y], half_sum, r[e].y * scale);
        if (row + 1 < rows) g.part[y + n] = (float)fma((double)g.field[y + n], half_sum, r[e].x * scale);
    }
}

// ------------------------------------------------------------------------- launchers

void fft_axis(int len, FftAxis& ax) {
    ax.n = len;
    ax.nrad = 0;
    int m = len;
    for (int r : {8, 4, 2, 3, 5})
        while (m % r == 0) {
            ax.rad[ax.nrad++] = (unsigned char)r;
            m /= r;
        }
}

// Lines of `len` points per block: about 1024 points (2 x 16 KB of shared memory and room for
// three blocks per SM), at most 16, at least 4 adjacent columns (64 bytes) of a strided axis.
int fft_lines_per_block(int len, bool strided) {
    int L = 1024 / len;
    if (L > 16) L = 16;
    const int least = strided ? (len > 2048 ? 1 : (len > 1024 ? 2 : 4)) : 1;
    return L < least ? least : L;
}

namespace {
int win_pairs(const FftArgs& g) { return ((g.n0 > 1 ? (g.P0 + 1) * (2 * g.P1 + 1) : g.P1 + 1) + 1) / 2; }
}

// The window's rows and planes are few: fewer lines a block, so that every SM has one (128^3, +-24:
// its four launches 80 us together with the field's 8 lines a block, 64 so).
void fft_window_lines(FftArgs& g) {
    g.Lv = std::max(1, std::min(g.Lx, win_pairs(g) / SMS));
    g.Lw = g.Ly;
    if (g.Lw > 4 && (int64_t)((g.nh + g.Lw - 1) / g.Lw) * (g.P0 + 1) < 2 * SMS) g.Lw = 4;
}

int fft_row_blocks(const FftArgs& g) { return (int)(((int64_t)g.n0 * g.n1 + 1) / 2 + g.Lx - 1) / g.Lx; }

namespace {
size_t row_smem(const FftArgs& g) { return (size_t)2 * g.Lx * g.n2 * sizeof(double2); }
size_t y_smem(const FftArgs& g) { return (size_t)2 * g.Ly * g.n1 * sizeof(double2); }
size_t last_smem(const FftArgs& g, bool mul) {
    const size_t pts = (size_t)g.Ll * (g.n0 > 1 ? g.n0 : g.n1);
    return 2 * pts * sizeof(double2) + (mul ? pts * sizeof(double) : 0);
}
unsigned win_blocks(const FftArgs& g) { return (unsigned)((win_pairs(g) + g.Lv - 1) / g.Lv); }
unsigned win_y_blocks(const FftArgs& g) { return (unsigned)((g.nh + g.Lw - 1) / g.Lw) * (g.P0 + 1); }
size_t win_smem(const FftArgs& g) { return (size_t)2 * g.Lv * g.n2 * sizeof(double2); }
size_t win_y_smem(const FftArgs& g) { return (size_t)2 * g.Lw * g.n1 * sizeof(double2); }
unsigned last_blocks(const FftArgs& g) { return (unsigned)((g.nh + g.Ll - 1) / g.Ll) * (g.n0 > 1 ? g.n1 : 1); }
unsigned y_blocks(const FftArgs& g, int planes) { return (unsigned)((g.nh + g.Ly - 1) / g.Ly) * planes; }

// twiddles, rows and the middle axis of the field
void field_spectrum(const FftArgs& g, cudaStream_t s) {
    const int longest = g.n0 > g.n1 ? (g.n0 > g.n2 ? g.n0 : g.n2) : (g.n1 > g.n2 ? g.n1 : g.n2);
    launch_dep(fft_twiddle_kernel, dim3((longest + 127) / 128, 3), 128, 0, s, g);
    launch_dep(fft_rows_kernel, (unsigned)fft_row_blocks(g), FFT_THREADS, row_smem(g), s, g);
    if (g.n0 > 1) launch_dep(fft_y_kernel<false>, y_blocks(g, g.n0), FFT_THREADS, y_smem(g), s, g);
}
}  // namespace

void launch_fft_descriptor(const FftArgs& g, cudaStream_t s) {
    field_spectrum(g, s);
    launch_dep(fft_last_kernel, last_blocks(g), FFT_THREADS, last_smem(g, false), s, g);
    if (g.n0 > 1) launch_dep(fft_win_y_kernel<true>, win_y_blocks(g), FFT_THREADS, win_y_smem(g), s, g);
    launch_dep(fft_desc_kernel, win_blocks(g), FFT_THREADS, win_smem(g), s, g);
}

// g.x_ready: the descriptor of the same call left X (and the twiddles) in place
void launch_fft_vjp(const FftArgs& g, cudaStream_t s) {
    if (!g.x_ready) field_spectrum(g, s);
    launch_dep(fft_coef_kernel, win_blocks(g), FFT_THREADS, win_smem(g), s, g);
    if (g.n0 > 1) launch_dep(fft_win_y_kernel<false>, win_y_blocks(g), FFT_THREADS, win_y_smem(g), s, g);
    launch_dep(fft_mul_kernel, last_blocks(g), FFT_THREADS, last_smem(g, true), s, g);
    if (g.n0 > 1) launch_dep(fft_y_kernel<true>, y_blocks(g, g.n0), FFT_THREADS, y_smem(g), s, g);
    launch_dep(fft_grad_kernel, (unsigned)fft_row_blocks(g), FFT_THREADS, row_smem(g), s, g);
}

void set_fft_attributes() {
    const void* ks[] = {(const void*)fft_rows_kernel,         (const void*)fft_y_kernel<false>,
                        (const void*)fft_y_kernel<true>,      (const void*)fft_last_kernel,
                        (const void*)fft_win_y_kernel<true>,  (const void*)fft_win_y_kernel<false>,
                        (const void*)fft_desc_kernel,         (const void*)fft_coef_kernel,
                        (const void*)fft_mul_kernel,          (const void*)fft_grad_kernel};
    for (const void* k : ks) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_DYN_SMEM);
}

}  // namespace dmcr
