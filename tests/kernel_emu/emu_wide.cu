// emu_wide.cu -- TEST HARNESS: the routing of pairs with large thresholds
// (the ring and the index kernels' whole routes) compiled for the host.  Not
// part of the library and never loaded by it.
#include <algorithm>
#include <cstdint>
#include <vector>

#include "ss_cws.cuh"
#include "ss_cwx.cuh"

using namespace ssk;

// The ring kernel's route for one pair, its lanes one after another.
template <class Sh>
static int ring_route(const uint32_t *q, const uint32_t *r, int m, int E)
{
    const int Ee = eff_threshold(m, E), lanes = Sh::LANES;
    std::vector<uint2> sm(Sh::WORDS / 2 + 1,
                          make_uint2(0xdeadbeefu, 0xdeadbeefu));
    uint2 *q2 = sm.data(), *r2 = q2 + Sh::QW + 1;
    std::vector<uint32_t> keep(2 * Sh::LW + 1, 0xdeadbeefu);
    RingStep s;
    s.q2 = q2;
    s.r2 = r2;
    s.q = q;
    s.r = r;
    s.m = m;
    s.w16 = (m + 15) >> 4;
    s.c = 0;
    int count = 0, qn = 0, rn = 0;
    for (;;) {
        qn = std::max(qn, std::max(s.c - Ee, 0) & ~(Sh::BP - 1));
        rn = std::max(rn, s.c & ~(Sh::BP - 1));
        for (; ring_room(qn, m, s.c - Ee, Sh::QB, Sh::BP); qn += Sh::BP)
            for (int t = 0; t < lanes; ++t)
                ring_load<Sh::QW, Sh::BP>(q2, q, s.w16, qn, t, lanes);
        for (; ring_room(rn, m, s.c, Sh::RB, Sh::BP); rn += Sh::BP)
            for (int t = 0; t < lanes; ++t)
                ring_load<Sh::RW, Sh::BP>(r2, r, s.w16, rn, t, lanes);
        const int until = std::min(ring_until(qn, m, Ee + kRingAhead),
                                   ring_until(rn, m, kRingAhead));
        if (until <= s.c)
            return -1001;  // no step would be made
        while (s.c < until) {
            ring_window<Sh::RW>(r2, s.c, s.rlo, s.rhi);
            s.lo = std::max(s.c - Ee, 0);
            s.hi = std::min(s.c + Ee, m - 1);
            int best = 0;
            for (int t = 0; t < lanes; ++t) {
                int open;
                best = std::max(best, ring_lane<Sh>(s, t, keep.data(), 2,
                                                    open));
                if (open < 0)
                    continue;
                const int lim = m - std::max(open, s.c);
                int all = 32;
                for (int k = 0; k < lanes && all == 32 + 32 * k; ++k)
                    all += ring_match<Sh>(s, open, all);
                if (all == 32 + 32 * lanes && all < lim)
                    all = ring_far(s, open, all, lim);
                best = std::max(best, all);
            }
            if (best < 4) {
                best = 0;
                for (int i = s.lo >> 5; i <= s.hi >> 5; ++i)
                    best = std::max(best, prefix_word<Sh>(s, m - s.c, i));
            }
            if (sm.back().x != 0xdeadbeefu || keep.back() != 0xdeadbeefu)
                return -1000;  // written past the slice
            s.c += best + 1;
            count += s.c <= m ? 1 : 0;
            if (s.c >= m || count > E)
                return count;
        }
    }
}

extern "C" {

// The ring route with the shape of class rc.
int emu_ring(const uint32_t *q, const uint32_t *r, int m, int E, int rc)
{
    return rc == 0   ? ring_route<RingShape<512, 512, 128, 2>>(q, r, m, E)
           : rc == 1 ? ring_route<RingShape<1024, 1024, 256>>(q, r, m, E)
                     : ring_route<RingShape<2048, 1024, 256>>(q, r, m, E);
}

}  // extern "C"

// The index kernel's route for one pair, its threads one after another: the
// lookups of the next columns (and the tables they build) before the chain
// follows the columns before them, as the kernel may.
template <class Sh>
static int route(uint32_t *tabs, const uint32_t *q, const uint32_t *r, int m,
                 int E)
{
    const int Ee = eff_threshold(m, E), w16 = (m + 15) >> 4, nt = Sh::COLS;
    std::vector<int> col[2] = {std::vector<int>(nt), std::vector<int>(nt)};
    int built = 0, buf = 0, at = 0, c0 = -nt;
    IndexChain chain{0, 0, 0};
    for (;;) {
        const int last = std::min(at + nt - 1 + Ee, m - 1);
        built = std::max(built, std::max(at - Ee, 0) >> Sh::LOGBS);
        for (; at < m && built <= last >> Sh::LOGBS; ++built) {
            uint32_t *tab = tabs + (built % Sh::NB) * Sh::SLOT;
            for (int t = 0; t < nt; ++t)
                table_clear<Sh>(tab, t, nt);
            for (int t = 0; t < nt; ++t)
                table_count<Sh>(tab, q, w16, m, built, t, nt);
            uint32_t sum = 0;
            for (int t = 0; t < nt; ++t) {
                const uint32_t own = table_sum<Sh>(tab, t, nt);
                table_prefix<Sh>(tab, sum, t, nt);
                sum += own;
            }
            for (int t = 0; t < nt; ++t)
                table_scatter<Sh>(tab, q, w16, m, built, t, nt);
        }
        for (int t = 0; t < nt; ++t)
            col[buf][t] = column_longest<Sh>(tabs, q, r, w16, m, Ee, at + t);
        chain_follow<Sh>(chain, col[buf ^ 1].data(), c0, nt, tabs, q, r, w16,
                         m, E, Ee, 0, 1);
        if (chain.done)
            return chain.count;
        c0 = at;
        at = std::max(at + nt, chain.c);
        buf ^= 1;
    }
}

extern "C" {

// The index route with the shape of class ic (3: a small shape of blocks of
// 16 starts, 8 columns at a time, whose ring turns often); a guard word
// after the tables.
int emu_index(const uint32_t *q, const uint32_t *r, int m, int E, int ic)
{
    using Small = IndexShape<2, 4, 4, 8>;
    static_assert(Small::max_e() == 16, "the small shape's threshold");
    std::vector<uint32_t> tabs(IndexShape2::WORDS + 1, 0xdeadbeefu);
    int n = -1, words = 0;
    switch (ic) {
    case 0: n = route<IndexShape0>(tabs.data(), q, r, m, E);
        words = IndexShape0::WORDS; break;
    case 1: n = route<IndexShape1>(tabs.data(), q, r, m, E);
        words = IndexShape1::WORDS; break;
    case 2: n = route<IndexShape2>(tabs.data(), q, r, m, E);
        words = IndexShape2::WORDS; break;
    default: n = route<Small>(tabs.data(), q, r, m, E);
        words = Small::WORDS; break;
    }
    return tabs[words] == 0xdeadbeefu ? n : -1000;
}

int emu_wide_class(int m, int E, int rw_max_e)
{
    TuneParams tp;
    tp.rw_max_e = rw_max_e;
    return class_of_tuned(m, E, tp);
}

// First ring, index and CTA class, the number of classes; the ring and index
// classes' E bounds.
int emu_class_table(int what, int c)
{
    switch (what) {
    case 0: return kFirstRing;
    case 1: return kFirstIndex;
    case 2: return kFirstCta;
    case 3: return kClasses;
    case 4: return ring_max_e(c);
    case 5: return index_max_e(c);
    default: return -1;
    }
}

}  // extern "C"
