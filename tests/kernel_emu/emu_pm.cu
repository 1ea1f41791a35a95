// emu_pm.cu -- TEST HARNESS: pair-major packed pairs walked bit-sliced (the
// turn of a group's words, the sub-maze mode's walk over them, and the
// capped distance) compiled for the host.  Not part of the library and never
// loaded by it.
#include <algorithm>
#include <cstdint>
#include <utility>
#include <vector>

#include "ss_pm.cuh"
#include "ss_sliced.cuh"

using namespace ssk;

namespace {

// One group's region of a side, as pm_stage fills it (n pairs from p0 on).
std::vector<uint32_t> region(const uint32_t *x, int64_t n, int64_t p0,
                             int w16)
{
    std::vector<uint32_t> out(pm_stride(w16), 0u);
    for (int i = 0; i < 32 && p0 + i < n; ++i)
        for (int c = 0; c < w16; ++c)
            out[pm_place(c, i)] = x[(p0 + i) * w16 + c];
    pm_turn(out.data(), w16);
    return out;
}

template <int E>
void one(const uint32_t *q, const uint32_t *r, int64_t n, int m, int what,
         int t, int y, int32_t *out)
{
    const int w16 = (m + 15) / 16;
    const SlicedEdges<E> ed(m);
    constexpr int WW = SlicedShape<E>::WW;
    std::vector<uint32_t> vtab(std::max(ed.rows(), 1) * WW);
    for (int i = 0; i < ed.rows() * WW; ++i)
        vtab[i] = SlicedEdges<E>::valid(ed.block_of(i / WW), i % WW, m);
    for (int64_t p0 = 0; p0 < n; p0 += 32) {
        const auto a = region(q, n, p0, w16), b = region(r, n, p0, w16);
        const PmSrc src{a.data(), b.data()};
        const int np = (int)std::min<int64_t>(32, n - p0);
        const uint32_t pad = np >= 32 ? 0u : 0xffffffffu << np;
        SlicedCount<E> cnt;
        if (what == 0)
            sliced_walk<E>(src, m, pad, cnt, vtab.data(), 1u,
                           SlicedSubMaze<E>(t, y));
        else
            ed_walk<E>(src, m, pad, cnt);
        uint32_t cb[SlicedShape<E>::NB];
        cnt.bits(cb);
        for (int i = 0; i < np; ++i)
            out[p0 + i] = sliced_count<E>(cb, i);
    }
}

template <int... Es>
void dispatch(int E, const uint32_t *q, const uint32_t *r, int64_t n, int m,
              int what, int t, int y, int32_t *out,
              std::integer_sequence<int, Es...>)
{
    ((E == Es ? (one<Es>(q, r, n, m, what, t, y, out), 0) : 0), ...);
}

}  // namespace

extern "C" {

// what: 0 sub-maze mode, 1 capped distance; out: the obstacles or distances
// of n fixed-stride packed pairs.
void emu_pm(const uint32_t *q, const uint32_t *r, int64_t n, int m, int E,
            int what, int t, int y, int32_t *out)
{
    dispatch(E, q, r, n, m, what, t, y, out,
             std::make_integer_sequence<int, 32>{});
}

void emu_transpose(uint32_t *a)
{
    uint32_t x[32];
    for (int i = 0; i < 32; ++i)
        x[i] = a[i];
    transpose32(x);
    for (int i = 0; i < 32; ++i)
        a[i] = x[i];
}

}  // extern "C"
