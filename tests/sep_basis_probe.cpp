// Host-only check of the separable path's tables (paper_2103_09686_gb300/csrc/sep_basis.cpp): for
// every range of the slope given as argument, the pairs F(u, v) = f((u + v) / 2)^2 that the FP32
// tables give, evaluated as the device does, against FP64.  Prints one line per range:
//   pairs, F(0, 0), largest |error| / (1e-5 F + 1e-9) for u, v in [0, 1], the same from 0 to the end
#include <math.h>
#include <stdio.h>
#include <stdlib.h>

#include <algorithm>
#include <vector>

#include "sep_basis.h"

int main(int argc, char** argv) {
    const double alpha = argc > 1 ? atof(argv[1]) : 10.0;
    const double s0 = 1.0 / (1.0 + exp(0.75 * alpha)), s1 = 1.0 / (1.0 + exp(-0.25 * alpha));
    const double c1 = 1.0 / (s1 - s0), c3 = -c1 * s0;
    auto F = [&](double t) {
        const double f = c1 / (1.0 + exp(-alpha * (0.5 * t - 0.75))) + c3;
        return f * f;
    };
    const auto b = dmcr::sep_basis((float)alpha);
    for (int k = 0; k < b->ntier; ++k) {
        const dmcr::SepTier& t = b->tier[k];
        std::vector<float> M;
        for (int i = 0; i <= 400; ++i) M.push_back((float)i / 400.f);
        const size_t unit = M.size();
        for (int i = 0; i <= 400; ++i) M.push_back(t.hi * (float)i / 400.f);
        std::vector<std::vector<float>> q;
        for (float m : M) {
            const float y = (float)dmcr::SEP_SEG * m;
            const int sg = std::min(std::max((int)rintf(y) - t.seg0, 0), t.nseg - 1);
            const float u = y - (float)(sg + t.seg0);
            std::vector<float> f;
            for (int p = 0; p < t.npair; ++p) {
                float x = 0.f, z = 0.f;
                for (int e = t.nc - 1; e >= 0; --e) {
                    const dmcr::SepCoef& c = b->coef[t.coef + ((size_t)e * t.npair + p) * t.nseg + sg];
                    x = fmaf(x, u, c.x);
                    z = fmaf(z, u, c.y);
                }
                f.push_back(x);
                f.push_back(z);
            }
            q.push_back(f);
        }
        double zero = 0.0, rel = 0.0, worst = 0.0;
        for (size_t i = 0; i < M.size(); ++i)
            for (size_t j = 0; j <= i; ++j) {
                double s = F(M[i]) + F(M[j]);
                for (int p = 0; p < t.npair; ++p)
                    s += (p < t.npos ? 1.0 : -1.0) * ((double)q[i][2 * p] * q[j][2 * p] + (double)q[i][2 * p + 1] * q[j][2 * p + 1]);
                const double want = F((double)M[i] + M[j]), err = fabs(s - want);
                worst = std::max(worst, err / (1e-5 * want + 1e-9));
                if (i < unit) rel = worst;
                if (i == 0 && j == 0) zero = s;
            }
        printf("%d %g %g %g\n", t.npair, zero, rel, worst);
    }
    return 0;
}
