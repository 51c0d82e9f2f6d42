// The value expansion of the separable path (sep.cu): plain C++ with no CUDA dependency, so that a
// host-only program can build the tables and check them.
#pragma once
#include <memory>
#include <vector>

namespace dmcr {

constexpr int SEP_TIERS = 6;        // value ranges with a basis of their own; tier SEP_TIERS: direct kernels
constexpr int SEP_MAX_PAIRS = 28;   // packed pairs of features of one basis at most
constexpr int SEP_SEG = 8;          // segments of the value range per unit
constexpr int SEP_MAX_NC = 14;      // coefficients of a feature in one segment at most
// Fields (any one phase) whose largest value stays below this are left to the direct kernels:
// their pairs are small against the rounding of the features (see build_tier).
constexpr float SEP_WEAK = 0.5f;

struct SepTier {
    float lo, hi;
    int seg0, nseg, nc;       // first segment, segments, coefficients per segment
    int npair, npos;          // packed pairs of features, the first npos of them with s = +1
    int coef;                 // offset of this tier's coefficients
};

struct SepCoef {
    float x, y;               // features 2 p and 2 p + 1
};

struct SepBasis {
    float alpha = 0.f;
    int ntier = 0;
    SepTier tier[SEP_TIERS] = {};
    std::vector<SepCoef> coef;
};

// the basis of one alpha (kept: the last few)
std::shared_ptr<const SepBasis> sep_basis(float alpha);

}  // namespace dmcr
