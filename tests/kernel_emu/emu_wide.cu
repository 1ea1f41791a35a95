// emu_wide.cu -- TEST HARNESS: the routing of pairs with large thresholds
// (the team kernel's word step and the index kernel's whole route) compiled
// for the host.  Not part of the library and never loaded by it.
#include <algorithm>
#include <cstdint>
#include <vector>

#include "ss_cwt.cuh"
#include "ss_cwx.cuh"

using namespace ssk;

extern "C" {

// The team kernel's loop for one pair, its lanes one after another.
int emu_team(const uint32_t *q, const uint32_t *r, int m, int E, int lanes)
{
    const int Ee = eff_threshold(m, E);
    const TeamLayout L = TeamLayout::of(m);
    std::vector<uint32_t> sm(L.words() + 1, 0xdeadbeefu);
    for (int t = 0; t < lanes; ++t)
        team_stage(sm.data(), L, q, r, m, t, lanes);
    if (sm.back() != 0xdeadbeefu)
        return -1000;  // staged past the slice
    int c = 0, count = 0;
    for (;;) {
        const uint32_t *r2 = sm.data() + 4 * L.PW + L.QW;
        const uint32_t rw = code_window(r2, c), rw2 = code_window(r2, c + 16);
        int o[4];
        for (int d = 0; d < 4; ++d)
            o[d] = (int)((rw >> (2 * d)) & 3u) * L.PW;
        const int lo = std::max(c - Ee, 0), hi = std::min(c + Ee, m - 1);
        const bool tail = c + 4 > m;
        int pstar = -1;
        for (int t = 0; t < lanes; ++t) {
            const int i = std::min((lo >> 5) + t, L.PW - 1);
            const uint32_t range = start_range(i, lo, hi);
            // a team with columns left may step beside one without
            const int a = team_word<true>(sm.data(), L, m, c, rw, rw2, o, i,
                                          range);
            if (!tail && a != team_word<false>(sm.data(), L, m, c, rw, rw2, o,
                                               i, range))
                return -1001;
            pstar = std::max(pstar, a);
        }
        if (pstar >= m)
            return count;
        ++count;
        if (count > E || pstar + 1 >= m)
            return count;
        c = pstar + 1;
    }
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

// The index route with the shape of class ic (4: a small shape of blocks of
// 16 starts, 8 columns at a time, whose ring turns often); a guard word
// after the tables.
int emu_index(const uint32_t *q, const uint32_t *r, int m, int E, int ic)
{
    using Small = IndexShape<2, 4, 4, 8>;
    static_assert(Small::max_e() == 16, "the small shape's threshold");
    std::vector<uint32_t> tabs(IndexShape3::WORDS + 1, 0xdeadbeefu);
    int n = -1, words = 0;
    switch (ic) {
    case 0: n = route<IndexShape0>(tabs.data(), q, r, m, E);
        words = IndexShape0::WORDS; break;
    case 1: n = route<IndexShape1>(tabs.data(), q, r, m, E);
        words = IndexShape1::WORDS; break;
    case 2: n = route<IndexShape2>(tabs.data(), q, r, m, E);
        words = IndexShape2::WORDS; break;
    case 3: n = route<IndexShape3>(tabs.data(), q, r, m, E);
        words = IndexShape3::WORDS; break;
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

// First team, index and CTA class; a team class's lanes, m bound and E
// bound; an index class's E bound.
int emu_class_table(int what, int c)
{
    switch (what) {
    case 0: return kFirstTeam;
    case 1: return kFirstIndex;
    case 2: return kFirstCta;
    case 3: return team_lanes(team_width_of(c));
    case 4: return team_mbound(c);
    case 5: return team_max_e(team_width_of(c));
    case 6: return index_max_e(c);
    case 7: return kClasses;
    default: return -1;
    }
}

}  // extern "C"
