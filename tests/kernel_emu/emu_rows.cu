// emu_rows.cu -- TEST HARNESS: the route of the ring kernel that a warp takes
// alone, what hands a pair over to it and how pairs are dealt to warps,
// compiled for the host.  Not part of the library and never loaded by it.
#include <algorithm>
#include <cstdint>
#include <vector>

#include "ss_cws.cuh"

using namespace ssk;

static const uint32_t kGuard = 0xdeadbeefu;

// The route of a warp with its lanes one after another; -1000: no progress,
// or a write past the rings.
template <class Sh>
static int warp_rows(const uint32_t *q, const uint32_t *r, int m, int E)
{
    const int Ee = eff_threshold(m, E);
    std::vector<uint2> x(Sh::WORDS / 2 + 1, make_uint2(kGuard, kGuard));
    uint2 *q2 = x.data(), *r2 = q2 + Sh::QW + 1;
    RingStep s;
    s.q2 = q2;
    s.r2 = r2;
    s.q = q;
    s.r = r;
    s.m = m;
    s.w16 = (m + 15) >> 4;
    s.c = 0;
    int qn = 0, rn = 0, count = 0;
    for (;;) {
        qn = std::max(qn, std::max(s.c - Ee, 0) & ~(Sh::BP - 1));
        rn = std::max(rn, s.c & ~(Sh::BP - 1));
        for (; ring_room(qn, m, s.c - Ee, Sh::QB, Sh::BP); qn += Sh::BP)
            for (int t = 0; t < 32; ++t)
                ring_load<Sh::QW, Sh::BP>(q2, q, s.w16, qn, t, 32);
        for (; ring_room(rn, m, s.c, Sh::RB, Sh::BP); rn += Sh::BP)
            for (int t = 0; t < 32; ++t)
                ring_load<Sh::RW, Sh::BP>(r2, r, s.w16, rn, t, 32);
        const int until = std::min(ring_until(qn, m, Ee + Sh::AHEAD),
                                   ring_until(rn, m, Sh::AHEAD));
        if (until <= s.c)
            return -1000;
        while (s.c < until) {
            ring_window<Sh::RW>(r2, s.c, s.rlo, s.rhi);
            s.lo = std::max(s.c - Ee, 0);
            s.hi = std::min(s.c + Ee, m - 1);
            int best = 0;
            bool many = false;
            for (int t = 0; t < 32; ++t)
                best = std::max(best, rows_step<Sh>(s, t, 1024, many));
            if (best < 4) {
                best = 0;
                for (int i = s.lo >> 5; i <= s.hi >> 5; ++i)
                    best = std::max(best, prefix_word<Sh>(s, m - s.c, i));
            }
            if (x.back().x != kGuard)
                return -1000;
            s.c += best + 1;
            count += s.c <= m ? 1 : 0;
            if (s.c >= m || count > E)
                return count;
        }
    }
}

// The column at which a team of the largest ring class hands the pair over
// to its warp, or -1 if it routes it to the end.
static int handed_over(const uint32_t *q, const uint32_t *r, int m, int E)
{
    using Sh = RingShape<2048, 1024, 256>;
    const int Ee = eff_threshold(m, E);
    std::vector<uint2> x(Sh::WORDS / 2);
    std::vector<uint32_t> keep(Sh::LW);
    uint2 *q2 = x.data(), *r2 = q2 + Sh::QW + 1;
    RingStep s{q2, r2, q, r, (m + 15) >> 4, m, 0, 0, 0, 0u, 0u};
    int count = 0, work[Sh::LANES] = {}, qn = 0, rn = 0;
    while (s.c < m && count <= E) {
        qn = std::max(qn, std::max(s.c - Ee, 0) & ~(Sh::BP - 1));
        rn = std::max(rn, s.c & ~(Sh::BP - 1));
        for (; ring_room(qn, m, s.c - Ee, Sh::QB, Sh::BP); qn += Sh::BP)
            for (int t = 0; t < Sh::LANES; ++t)
                ring_load<Sh::QW, Sh::BP>(q2, q, s.w16, qn, t, Sh::LANES);
        for (; ring_room(rn, m, s.c, Sh::RB, Sh::BP); rn += Sh::BP)
            for (int t = 0; t < Sh::LANES; ++t)
                ring_load<Sh::RW, Sh::BP>(r2, r, s.w16, rn, t, Sh::LANES);
        ring_window<Sh::RW>(r2, s.c, s.rlo, s.rhi);
        s.lo = std::max(s.c - Ee, 0);
        s.hi = std::min(s.c + Ee, m - 1);
        int best = 0;
        for (int t = 0; t < Sh::LANES; ++t) {
            int open;
            best = std::max(best, ring_lane<Sh>(s, t, keep.data(), 1, open,
                                                work[t]));
            if (open >= 0)
                best = std::max(best, ring_follow<Sh>(
                                          s, open, 32,
                                          m - std::max(open, s.c)));
        }
        s.c += best + 1;
        ++count;
        for (int t = 0; t < Sh::LANES; ++t)
            if (work[t] > ring_work_limit(s.c, count))
                return s.c;
    }
    return -1;
}

extern "C" {

// All rows by a warp.
int emu_rows(const uint32_t *q, const uint32_t *r, int m, int E, int which)
{
    return which == 0 ? warp_rows<WarpShape>(q, r, m, E) : -1;
}

int emu_rows_max_e(int which)
{
    return which == 0 ? WarpShape::max_e() : -1;
}

int emu_handed_over(const uint32_t *q, const uint32_t *r, int m, int E)
{
    return handed_over(q, r, m, E);
}

int emu_first_pair(int b, int grid, int sms)
{
    return first_pair(b, grid, sms);
}

}  // extern "C"
