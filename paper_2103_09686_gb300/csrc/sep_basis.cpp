// Basis of the separable path (sep.cu), built on the host in FP64.  Paper: arXiv 2103.09686,
// Sec. 3.2.2-3.2.4.
//
// The pair function F(u, v) = f((u + v) / 2)^2 is smooth on the bounded range of a relaxed field,
// so its integral operator has rapidly decaying eigenvalues.  The background M = 0 is taken out
// first: F(0, 0) = 0, and with phi(u) = F(u, 0)
//     F(u, v) = phi(u) + phi(v) + sum_k s_k q_k(u) q_k(v),   s_k = +-1,  q_k(0) = 0 exactly,
// so that a descriptor scales with the share of a medium that is not background, as its pairs
// do.  (With the background left in the features, sum_k s_k p_k(0)^2 = 0 has to come out of terms of
// order 1 rounded to FP32: the entries of a 1 % medium in the widest range were off by 1e-3.)
// phi needs no transform: it enters a descriptor by its mean alone.  (The device goes on from there to
// features that vanish at the mean of a grey field, sep.cu.)
//
// The same holds, less sharply, for dark values: F(0.3, 0.3) is 1e-4.  The eigenfunctions are
// therefore taken of F - phi - phi weighted by 1 / (w(u) w(v)), w(u)^2 = f(u)^2 + delta^2 (and
// growing again below 0, where F is small but its values with bright partners are not), which makes a
// feature about as small as the pairs it serves: the sum of q_k(0.3)^2 falls from 0.4 to about
// 0.02 in the wide ranges, with as many pairs as without the weight.
#include "sep_basis.h"

#include <math.h>

#include <algorithm>
#include <mutex>

namespace dmcr {

namespace {

struct PairFn {
    double a, c1, c3;
    explicit PairFn(double alpha) : a(alpha) {
        const double s0 = 1.0 / (1.0 + exp(0.75 * a)), s1 = 1.0 / (1.0 + exp(-0.25 * a));
        c1 = 1.0 / (s1 - s0);
        c3 = -c1 * s0;
    }
    double f(double t) const { return c1 / (1.0 + exp(-a * (0.5 * t - 0.75))) + c3; }
    double F(double t) const { const double v = f(t); return v * v; }          // t = u + v
    double Fu(double t) const {
        const double s = 1.0 / (1.0 + exp(-a * (0.5 * t - 0.75)));
        return (c1 * s + c3) * c1 * a * s * (1.0 - s);
    }
    double weight(double u, double delta) const {
        const double below = u < 0.0 ? 0.2 * u : 0.0;
        return sqrt(F(2.0 * u) + delta * delta + below * below);
    }
};

// Symmetric eigenproblem by cyclic Jacobi rotations (Golub & Van Loan, Matrix Computations,
// Sec. 8.5): A (n x n) becomes diagonal, V holds the eigenvectors in its columns.
void jacobi_eigen(std::vector<double>& A, std::vector<double>& V, int n) {
    V.assign((size_t)n * n, 0.0);
    for (int i = 0; i < n; ++i) V[(size_t)i * n + i] = 1.0;
    for (int sweep = 0; sweep < 30; ++sweep) {
        double off = 0.0, dia = 0.0;
        for (int i = 0; i < n; ++i)
            for (int j = 0; j < n; ++j) (i == j ? dia : off) += A[(size_t)i * n + j] * A[(size_t)i * n + j];
        if (off <= 1e-30 * dia) break;
        for (int p = 0; p < n; ++p)
            for (int q = p + 1; q < n; ++q) {
                const double apq = A[(size_t)p * n + q];
                if (apq == 0.0) continue;
                const double th = (A[(size_t)q * n + q] - A[(size_t)p * n + p]) / (2.0 * apq);
                const double t = (th >= 0 ? 1.0 : -1.0) / (fabs(th) + sqrt(th * th + 1.0));
                const double c = 1.0 / sqrt(t * t + 1.0), s = t * c;
                for (int k = 0; k < n; ++k) {
                    const double x = A[(size_t)k * n + p], y = A[(size_t)k * n + q];
                    A[(size_t)k * n + p] = c * x - s * y;
                    A[(size_t)k * n + q] = s * x + c * y;
                }
                for (int k = 0; k < n; ++k) {
                    const double x = A[(size_t)p * n + k], y = A[(size_t)q * n + k];
                    A[(size_t)p * n + k] = c * x - s * y;
                    A[(size_t)q * n + k] = s * x + c * y;
                }
                for (int k = 0; k < n; ++k) {
                    const double x = V[(size_t)k * n + p], y = V[(size_t)k * n + q];
                    V[(size_t)k * n + p] = c * x - s * y;
                    V[(size_t)k * n + q] = s * x + c * y;
                }
            }
    }
}

// What one tier is built to: largest errors of F and dF/du over its range, absolute and in units
// of w(u) w(v).
struct TierTol {
    double delta, F, Fu, wF, wFu;
};

enum TierResult { TIER_OK, TIER_ROUNDED, TIER_NONE };

// One tier: eigenfunctions on the range of the segments k0 .. k1 (segment k holds the values
// within half a segment of k / SEP_SEG; k0 <= 0 <= k1), discretised at Chebyshev nodes, as one
// short polynomial per segment.  TIER_NONE when SEP_MAX_PAIRS packed pairs, or polynomials of
// SEP_MAX_NC coefficients, do not reach the tolerances (a smaller delta would need more of both).
// TIER_ROUNDED when the tables, rounded to FP32 as the device reads them, give a pair of values from
// 0 up further off than 1e-5 F + 1e-9 -- what an entry of the descriptor may be off; a medium of two
// values consists of few such pairs -- or any pair further off than 1e-5.
TierResult build_tier(const PairFn& fn, int k0, int k1, const TierTol& tol, SepTier& t, std::vector<SepCoef>& coef) {
    const double lo = (k0 - 0.5) / SEP_SEG, hi = (k1 + 0.5) / SEP_SEG;
    const double mid = 0.5 * (lo + hi), half = 0.5 * (hi - lo);
    // nodes: the degree grows with the range measured in widths of the sigmoid
    const int n = (int)std::min(160.0, std::max(48.0, 24.0 + 2.6 * (hi - lo) * fn.a));
    std::vector<double> ct(4 * n);                       // cos(pi m / (2 n))
    for (int m = 0; m < 4 * n; ++m) ct[m] = cos(M_PI * m / (2 * n));
    std::vector<double> x(n), w(n), phi(n);              // nodes, their weights and background pairs
    for (int i = 0; i < n; ++i) {
        x[i] = mid + half * ct[2 * i + 1];
        w[i] = fn.weight(x[i], tol.delta);
        phi[i] = fn.F(x[i]);
    }
    std::vector<double> A((size_t)n * n);
    for (int i = 0; i < n; ++i)
        for (int j = 0; j < n; ++j) A[(size_t)i * n + j] = (fn.F(x[i] + x[j]) - phi[i] - phi[j]) / (w[i] * w[j] * n);
    // numerical range of A: Gram-Schmidt on its columns, largest residual first, each
    // direction orthogonalised twice
    const int rmax = std::min(n, 2 * SEP_MAX_PAIRS + 8);
    std::vector<double> W(A), Q;                          // W: residual columns (A is symmetric: rows); Q: r rows
    int r = 0;
    double first = 0.0;
    for (; r < rmax; ++r) {
        int best = 0;
        double bestn = -1.0;
        for (int j = 0; j < n; ++j) {
            double s = 0.0;
            for (int i = 0; i < n; ++i) s += W[(size_t)j * n + i] * W[(size_t)j * n + i];
            if (s > bestn) bestn = s, best = j;
        }
        if (r == 0) first = bestn;
        if (!(bestn > 1e-28 * first)) break;
        std::vector<double> q(W.begin() + (size_t)best * n, W.begin() + (size_t)(best + 1) * n);
        for (int k = 0; k < r; ++k) {
            double d = 0.0;
            for (int i = 0; i < n; ++i) d += q[i] * Q[(size_t)k * n + i];
            for (int i = 0; i < n; ++i) q[i] -= d * Q[(size_t)k * n + i];
        }
        double nn = 0.0;
        for (double v : q) nn += v * v;
        nn = 1.0 / sqrt(nn);
        for (double& v : q) v *= nn;
        for (int j = 0; j < n; ++j) {
            double d = 0.0;
            for (int i = 0; i < n; ++i) d += q[i] * W[(size_t)j * n + i];
            for (int i = 0; i < n; ++i) W[(size_t)j * n + i] -= d * q[i];
        }
        Q.insert(Q.end(), q.begin(), q.end());
    }
    // A restricted to it, and its eigenvectors
    std::vector<double> AQ((size_t)r * n), B((size_t)r * r), V;
    for (int k = 0; k < r; ++k)
        for (int i = 0; i < n; ++i) {
            double s = 0.0;
            for (int j = 0; j < n; ++j) s += A[(size_t)i * n + j] * Q[(size_t)k * n + j];
            AQ[(size_t)k * n + i] = s;
        }
    for (int k = 0; k < r; ++k)
        for (int m = 0; m < r; ++m) {
            double s = 0.0;
            for (int i = 0; i < n; ++i) s += Q[(size_t)m * n + i] * AQ[(size_t)k * n + i];
            B[(size_t)k * r + m] = s;
        }
    for (int k = 0; k < r; ++k)
        for (int m = 0; m < k; ++m)
            B[(size_t)k * r + m] = B[(size_t)m * r + k] = 0.5 * (B[(size_t)k * r + m] + B[(size_t)m * r + k]);
    jacobi_eigen(B, V, r);
    std::vector<int> ord(r);
    for (int i = 0; i < r; ++i) ord[i] = i;
    std::stable_sort(ord.begin(), ord.end(),
                     [&](int a, int b) { return fabs(B[(size_t)a * r + a]) > fabs(B[(size_t)b * r + b]); });
    // Chebyshev coefficients of sqrt(|lambda_k| n) w v_k
    auto series = [&](int k) {
        std::vector<double> v(n, 0.0), c(n);
        for (int m = 0; m < r; ++m)
            for (int i = 0; i < n; ++i) v[i] += V[(size_t)m * r + ord[k]] * Q[(size_t)m * n + i];
        for (int i = 0; i < n; ++i) v[i] *= w[i];
        const double sc = sqrt(fabs(B[(size_t)ord[k] * r + ord[k]]) * n);
        for (int j = 0; j < n; ++j) {
            double s = 0.0;
            for (int i = 0; i < n; ++i) s += v[i] * ct[(int)((int64_t)j * (2 * i + 1) % (4 * n))];
            c[j] = s * sc * (j == 0 ? 1.0 : 2.0) / n;
        }
        return c;
    };
    constexpr int GRID = 97;
    std::vector<double> E((size_t)GRID * GRID), D((size_t)GRID * GRID), limF(E.size()), limD(E.size());
    auto gx = [&](int i) { return -1.0 + 2.0 * i / (GRID - 1); };
    for (int i = 0; i < GRID; ++i)
        for (int j = 0; j < GRID; ++j) {
            const double u = mid + half * gx(i), v = mid + half * gx(j);
            const double ww = fn.weight(u, tol.delta) * fn.weight(v, tol.delta);
            const size_t o = (size_t)i * GRID + j;
            E[o] = fn.F(u + v) - fn.F(u) - fn.F(v);
            D[o] = fn.Fu(u + v) - fn.Fu(u);
            limF[o] = std::min(tol.F, tol.wF * ww);
            limD[o] = std::min(tol.Fu, tol.wFu * ww);
        }
    std::vector<std::vector<double>> pos, neg;
    bool ok = false;
    for (int k = 0; k < r; ++k) {
        const bool plus = B[(size_t)ord[k] * r + ord[k]] > 0.0;
        std::vector<std::vector<double>>& side = plus ? pos : neg;
        // once accurate, further terms are taken only while they fill a half-empty pair
        if (ok && side.size() % 2 == 0) break;
        if ((int)((pos.size() + 1) / 2 + (neg.size() + 1) / 2) + (side.size() % 2 == 0) > SEP_MAX_PAIRS) break;
        const std::vector<double> c = series(k);
        side.push_back(c);
        std::vector<double> p(GRID), dp(GRID);
        for (int i = 0; i < GRID; ++i) {
            const double xx = gx(i);
            double T0 = 1.0, T1 = xx, U0 = 1.0, U1 = 2.0 * xx, s = c[0] + c[1] * xx, d = c[1];
            for (int j = 2; j < n; ++j) {
                const double T2 = 2.0 * xx * T1 - T0;
                s += c[j] * T2;
                d += c[j] * j * U1;          // T_j' = j U_{j-1}
                T0 = T1, T1 = T2;
                const double U2 = 2.0 * xx * U1 - U0;
                U0 = U1, U1 = U2;
            }
            p[i] = s;
            dp[i] = d / half;
        }
        bool good = true;
        for (int i = 0; i < GRID; ++i)
            for (int j = 0; j < GRID; ++j) {
                const size_t o = (size_t)i * GRID + j;
                E[o] -= (plus ? 1.0 : -1.0) * p[i] * p[j];
                D[o] -= (plus ? 1.0 : -1.0) * dp[i] * p[j];
                good = good && fabs(E[o]) < limF[o] && fabs(D[o]) < limD[o];
            }
        ok = ok || good;
    }
    if (!ok) return TIER_NONE;
    // local polynomials in u = SEP_SEG M - k, |u| <= 1/2: interpolation at SEP_MAX_NC + 4
    // Chebyshev points, cut where the rest is below the rounding of the largest terms
    constexpr int m = SEP_MAX_NC + 4;
    const int nseg = k1 - k0 + 1, npos = (int)(pos.size() + 1) / 2, npair = npos + (int)(neg.size() + 1) / 2;
    std::vector<double> local((size_t)2 * npair * nseg * m, 0.0);       // [feature][segment][power]
    double at[m], dct[m][m], mono[m][m] = {};       // points, their cosines, powers of u of T_q(2 u)
    for (int i = 0; i < m; ++i) {
        at[i] = 0.5 * cos((i + 0.5) * M_PI / m);
        for (int q = 0; q < m; ++q) dct[q][i] = cos(q * (i + 0.5) * M_PI / m) * (q == 0 ? 1.0 : 2.0) / m;
    }
    mono[0][0] = 1.0;
    mono[1][1] = 2.0;
    for (int q = 2; q < m; ++q)
        for (int e = 0; e < m; ++e) mono[q][e] = (e > 0 ? 4.0 * mono[q - 1][e - 1] : 0.0) - mono[q - 2][e];
    int nc = 4;
    std::vector<double> T((size_t)m * n);            // T_q at the points of one segment
    for (int sg = 0; sg < nseg; ++sg) {
        for (int i = 0; i < m; ++i) {
            double* row = &T[(size_t)i * n];
            const double xx = ((k0 + sg + at[i]) / SEP_SEG - mid) / half;
            row[0] = 1.0;
            row[1] = xx;
            for (int q = 2; q < n; ++q) row[q] = 2.0 * xx * row[q - 1] - row[q - 2];
        }
        const double cut = 1e-8 * fn.weight((double)(k0 + sg) / SEP_SEG, tol.delta);
        for (int side = 0; side < 2; ++side)
            for (size_t k = 0; k < (side ? neg : pos).size(); ++k) {
                const std::vector<double>& c = (side ? neg : pos)[k];
                double* power = &local[(((side ? 2 * npos : 0) + k) * nseg + sg) * m];
                double y[m];
                for (int i = 0; i < m; ++i) {
                    double s[4] = {};
                    for (int q = 0; q + 4 <= n; q += 4)
                        for (int j = 0; j < 4; ++j) s[j] += c[q + j] * T[(size_t)i * n + q + j];
                    for (int q = n & ~3; q < n; ++q) s[0] += c[q] * T[(size_t)i * n + q];
                    y[i] = (s[0] + s[1]) + (s[2] + s[3]);
                }
                for (int q = 0; q <= SEP_MAX_NC; ++q) {
                    double ch = 0.0;
                    for (int i = 0; i < m; ++i) ch += y[i] * dct[q][i];
                    if (fabs(ch) > cut) nc = std::max(nc, q + 1);
                    if (q < SEP_MAX_NC)
                        for (int e = 0; e <= q; ++e) power[e] += ch * mono[q][e];
                }
                if (nc > SEP_MAX_NC) return TIER_NONE;
            }
    }
    // q_k = p_k - p_k(0): M = 0 is the centre of segment 0, where the constant becomes exactly 0
    for (int p = 0; p < 2 * npair; ++p) {
        const double zero = local[((size_t)p * nseg - k0) * m];
        for (int sg = 0; sg < nseg; ++sg) local[((size_t)p * nseg + sg) * m] -= zero;
    }
    t.lo = (float)lo;
    t.hi = (float)hi;
    t.seg0 = k0;
    t.nseg = nseg;
    t.nc = nc;
    t.npos = npos;
    t.npair = npair;
    t.coef = (int)coef.size();
    // coefficients [power][pair][segment] of the features (2p, 2p + 1)
    std::vector<SepCoef> table;
    for (int e = 0; e < nc; ++e)
        for (int p = 0; p < npair; ++p)
            for (int sg = 0; sg < nseg; ++sg)
                table.push_back({(float)local[((size_t)(2 * p) * nseg + sg) * m + e],
                                 (float)local[((size_t)(2 * p + 1) * nseg + sg) * m + e]});
    // the rounded tables, evaluated in FP32 as on the device: values from 0 to hi, then the whole range
    constexpr int UP = 401, ALL = 101;
    const int nf = 2 * npair;
    std::vector<double> q((size_t)(UP + ALL) * nf), M(UP + ALL), bg(UP + ALL);
    for (int i = 0; i < UP + ALL; ++i) {
        const float v = (float)(i < UP ? hi * i / (UP - 1) : lo + (hi - lo) * (i - UP) / (ALL - 1));
        const float y = (float)SEP_SEG * v;
        const int sg = std::min(std::max((int)lrintf(y) - k0, 0), nseg - 1);
        const float u = y - (float)(sg + k0);
        M[i] = v;
        bg[i] = fn.F(v);
        for (int p = 0; p < npair; ++p) {
            SepCoef s{0.f, 0.f};
            for (int e = nc - 1; e >= 0; --e) {
                const SepCoef& k = table[((size_t)e * npair + p) * nseg + sg];
                s = {fmaf(s.x, u, k.x), fmaf(s.y, u, k.y)};
            }
            q[(size_t)i * nf + 2 * p] = s.x;
            q[(size_t)i * nf + 2 * p + 1] = s.y;
        }
    }
    auto good = [&](int i, int j) {
        const double *a = &q[(size_t)i * nf], *b = &q[(size_t)j * nf];
        double plus = 0.0, minus = 0.0;
        for (int k = 0; k < 2 * npos; ++k) plus += a[k] * b[k];
        for (int k = 2 * npos; k < nf; ++k) minus += a[k] * b[k];
        const double F = fn.F(M[i] + M[j]);
        return fabs(bg[i] + bg[j] + plus - minus - F) <= (i < UP ? 1e-5 * F + 1e-9 : 1e-5);
    };
    for (int i = 0; i < UP; ++i)                     // equal values are the likeliest to fail
        if (!good(i, i)) return TIER_ROUNDED;
    for (int i = 0; i < UP + ALL; ++i)
        for (int j = i < UP ? 0 : UP; j <= i; ++j)
            if (!good(i, j)) return TIER_ROUNDED;
    coef.insert(coef.end(), table.begin(), table.end());
    return TIER_OK;
}

// The first range, [-1/16, 17/16], is a field between the phases with the overshoot of an optimiser
// step or two; the penalty weakens as the loss falls, so fields of long runs spread over the wider
// ones, up to [-2.3, 2.6] (measured over 3000 Adam steps: [-1.7, 1.9]).  A wider range needs more
// features: 7, 10, 14, 15, 19, 24 packed pairs at alpha = 10.
void build(SepBasis& b) {
    const PairFn fn((double)b.alpha);
    const int ranges[SEP_TIERS][2] = {{0, 8}, {-2, 10}, {-4, 12}, {-8, 13}, {-12, 16}, {-18, 20}};   // segments
    // Truncation below the FP32 rounding of a pair's value and derivative.  Of the weights, the
    // largest delta whose rounded tables are good: in the wide ranges 0.02 keeps grey fields with
    // a few bright pixels near 1e-6 (0.05, one pair less in some: 2e-6 .. 1e-5), at features of up to
    // 4 for values beyond 1; steeper slopes need smaller ones.  A range needs much the same as the
    // one before.
    const double deltas[] = {0.2, 0.05, 0.02, 0.014, 0.01, 0.007, 0.005};
    constexpr int ND = sizeof deltas / sizeof deltas[0];
    int d = 0;
    b.ntier = 0;
    b.coef.clear();
    for (int t = 0; t < SEP_TIERS; ++t) {
        TierResult res = TIER_ROUNDED;
        for (d = t == 0 ? 0 : std::max(2, d - 1); d < ND; ++d) {
            const double delta = deltas[d];
            const TierTol tol = t == 0 ? TierTol{delta, 5e-9, 7e-7, 1e-6, 1e-4} : TierTol{delta, 2e-8, 1e-6, 1e-6, 1e-5};
            res = build_tier(fn, ranges[t][0], ranges[t][1], tol, b.tier[t], b.coef);
            if (res != TIER_ROUNDED) break;
        }
        if (res != TIER_OK) break;
        b.ntier = t + 1;
    }
}

}  // namespace

std::shared_ptr<const SepBasis> sep_basis(float alpha) {
    // one build takes about 0.1 s: outside the lock, so that only callers of the same new alpha wait
    struct Entry {
        SepBasis basis;
        std::once_flag built;
    };
    static std::mutex mu;
    static std::vector<std::shared_ptr<Entry>>* cache = new std::vector<std::shared_ptr<Entry>>();
    constexpr size_t KEEP = 16;
    std::shared_ptr<Entry> e;
    {
        std::lock_guard<std::mutex> lk(mu);
        size_t i = 0;
        while (i < cache->size() && (*cache)[i]->basis.alpha != alpha) ++i;
        if (i == cache->size()) {
            auto fresh = std::make_shared<Entry>();
            fresh->basis.alpha = alpha;
            cache->push_back(fresh);
        }
        std::rotate(cache->begin(), cache->begin() + i, cache->begin() + i + 1);   // most recent first
        if (cache->size() > KEEP) cache->pop_back();
        e = cache->front();
    }
    std::call_once(e->built, [&] { build(e->basis); });
    return std::shared_ptr<const SepBasis>(e, &e->basis);
}

}  // namespace dmcr
