// Host-only check of the limit on a fused launch's blocks (paper_2103_09686_gb300/csrc/api.cu,
// prepare): the direct launches behind separable problems count as the others do.  Builds the tables
// of a batch whose direct kernels would need more than 2^31 - 1 blocks; nothing is launched and
// no device memory is touched.  Prints the blocks and the status; exits 1 unless it is refused.
#include "../paper_2103_09686_gb300/csrc/api.cu"

int main() {
    using namespace dmcr;
    dmcr_params p{};
    p.ndim = 3;
    p.n[0] = 64, p.n[1] = 2048, p.n[2] = 2048;
    p.window[0] = 32, p.window[1] = 64, p.window[2] = 32;
    p.levels = 1;
    p.alpha = 10.f;
    p.level_weight_exp = -1.f;
    Plan pl;
    if (validate_and_plan(&p, pl) != DMCR_OK || !pl.sep) return 2;
    constexpr int COUNT = 64;
    const double blocks = (double)pl.g[0].fwdTiles * pl.g[0].fwdGroupBlocks * COUNT;
    char* ws = reinterpret_cast<char*>(size_t(1) << 30);          // addresses only
    std::vector<Inst> in;
    for (int i = 0; i < COUNT; ++i) {
        Inst x = single(pl, ws);
        x.sc = nullptr;
        x.field = reinterpret_cast<const float*>(ws);
        x.desc = reinterpret_cast<float*>(ws);
        in.push_back(x);
    }
    Prepared P;
    const dmcr_status st = prepare(in, F_FWD, ws, size_t(1) << 40, 0, P);
    printf("%.3g blocks: status %d %s\n", blocks, (int)st, st != DMCR_OK ? dmcr_last_error() : "");
    return blocks > 2147483647.0 && st == DMCR_ENOTSUP ? 0 : 1;
}
