// emu_diag.cu -- TEST HARNESS: the distance kernel by diagonals (any threshold
// up to 511, a team of lanes per pair) compiled for the host.  Not part of
// the library and never loaded by it.
#include <cstdint>
#include <vector>

#include "ss_verify.cuh"

using namespace ssk;

// min(ED, E+1) by a team of nt lanes, taken in turn, with the arrays of a
// launch for thresholds up to top; -1000: written past them.
extern "C" int emu_diag(const uint32_t *q, const uint32_t *r, int m, int E,
                        int nt, int top)
{
    const int H = top / 2, W = 2 * H + 3, w16 = (m + 15) >> 4;
    const int guard = 0x5eadbeef;
    std::vector<int> F[2] = {std::vector<int>(W + 2, kEdNone),
                             std::vector<int>(W + 2, kEdNone)};
    for (auto &f : F)
        f.front() = f.back() = guard;
    F[0][H + 2] = ed_slide(q, r, w16, 0, 0, m);
    for (int e = 0;; ++e) {
        int ed;
        if (ed_ends(F[e & 1][H + 2], m, E, e, ed))
            return F[0].front() == guard && F[0].back() == guard &&
                           F[1].front() == guard && F[1].back() == guard
                       ? ed
                       : -1000;
        for (int t = nt - 1; t >= 0; --t)  // (no lane needs another's)
            ed_advance(q, r, w16, m, E, e, F[e & 1].data() + H + 2,
                       F[(e + 1) & 1].data() + H + 2, t, nt);
    }
}
