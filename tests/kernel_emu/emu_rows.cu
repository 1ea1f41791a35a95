// emu_rows.cu -- TEST HARNESS: the all-rows routes of the ring and the index
// kernels (a warp or a CTA per pair), what hands a pair over to them, the
// index' way back, and how pairs are dealt to warps, compiled for the host.  Not part of the library and never loaded by it.
#include <algorithm>
#include <cstdint>
#include <vector>

#include "ss_cws.cuh"
#include "ss_cwx.cuh"

using namespace ssk;

static const uint32_t kGuard = 0xdeadbeefu;

// Follow the chain by all rows with the lanes one after another, until its
// end or `calm` quiet stretches.  False: no progress, or a write past the slice.
template <class Sh>
static bool rows(IndexChain &chain, const uint32_t *q, const uint32_t *r,
                 int m, int E, int Ee, int calm, int dense)
{
    std::vector<uint2> x(Sh::WORDS / 2 + 1, make_uint2(kGuard, kGuard));
    uint2 *q2 = x.data(), *r2 = q2 + Sh::QW + 1;
    RingStep s;
    s.q2 = q2;
    s.r2 = r2;
    s.q = q;
    s.r = r;
    s.m = m;
    s.w16 = (m + 15) >> 4;
    s.c = chain.c;
    int qn = 0, rn = 0, quiet = 0;
    for (;;) {
        qn = std::max(qn, std::max(s.c - Ee, 0) & ~(Sh::BP - 1));
        rn = std::max(rn, s.c & ~(Sh::BP - 1));
        const int q0 = qn, r0 = rn;
        while (ring_room(qn, m, s.c - Ee, Sh::QB, Sh::BP))
            qn += Sh::BP;
        while (ring_room(rn, m, s.c, Sh::RB, Sh::BP))
            rn += Sh::BP;
        for (int t = 0; t < Sh::LANES; ++t) {
            ring_fill<Sh::QW>(q2, q, s.w16, q0, qn, t, Sh::LANES);
            ring_fill<Sh::RW>(r2, r, s.w16, r0, rn, t, Sh::LANES);
        }
        const int until = std::min({ring_until(qn, m, Ee + Sh::AHEAD),
                                    ring_until(rn, m, Sh::AHEAD),
                                    s.c + kRowsStretch});
        if (until <= s.c)
            return false;
        const int c0 = s.c, count0 = chain.count;
        bool many = false;
        while (s.c < until) {
            ring_window<Sh::RW>(r2, s.c, s.rlo, s.rhi);
            s.lo = std::max(s.c - Ee, 0);
            s.hi = std::min(s.c + Ee, m - 1);
            int best = 0;
            for (int t = 0; t < Sh::LANES; ++t)
                best = std::max(best, rows_step<Sh>(s, t, 32 * Sh::LANES,
                                                    many));
            if (best < 4) {
                best = 0;
                for (int i = s.lo >> 5; i <= s.hi >> 5; ++i)
                    best = std::max(best, prefix_word<Sh>(s, m - s.c, i));
            }
            if (x.back().x != kGuard)
                return false;
            s.c += best + 1;
            chain.count += s.c <= m ? 1 : 0;
            chain.c = s.c;
            chain.done = s.c >= m || chain.count > E;
            if (chain.done)
                return true;
        }
        quiet = many ? 0 : quiet + 1;
        if (quiet >= calm && s.c - c0 < dense * (chain.count - count0))
            return true;
    }
}

template <class Sh>
static int all_rows(const uint32_t *q, const uint32_t *r, int m, int E)
{
    IndexChain chain{0, 0, 0};
    return rows<Sh>(chain, q, r, m, E, eff_threshold(m, E), 1, 0)
               ? chain.count
                                                               : -1000;
}

// The index route of class C; turns: how often it went over to all rows.
template <int C>
static int index_rows(const uint32_t *q, const uint32_t *r, int m, int E,
                      int calm, int *turns)
{
    using Sh = typename IndexClass<C>::Shape;
    using Rows = typename IndexClass<C>::Rows;
    const int Ee = eff_threshold(m, E), w16 = (m + 15) >> 4, nt = Sh::COLS;
    std::vector<uint32_t> tabs(Sh::WORDS + 1, kGuard);
    std::vector<int> col[2] = {std::vector<int>(nt), std::vector<int>(nt)};
    const int STEPS = IndexClass<C>::STEPS, DENSE = nt / (2 * STEPS);
    int built = 0, buf = 0, at = 0, c0 = -nt, steps = 8 * STEPS, before = 0;
    IndexChain chain{0, 0, 0};
    bool all = (int64_t)Ee * kIndexSparse < m;
    *turns = 0;
    for (;;) {
        if (all) {
            ++*turns;
            const int c = chain.c;
            if (!rows<Rows>(chain, q, r, m, E, Ee, calm, DENSE) ||
                chain.c <= c)
                return -1001;
            if (chain.done)
                return chain.count;
            all = false;
            built = 0;
            std::fill(tabs.begin(), tabs.end() - 1, 0xdeadbeefu);
            steps = 8 * STEPS;
            before = chain.count;
            at = chain.c;
            c0 = at - nt;
        }
        const int last = std::min(at + nt - 1 + Ee, m - 1);
        built = std::max(built, std::max(at - Ee, 0) >> Sh::LOGBS);
        for (; at < m && built <= last >> Sh::LOGBS; ++built) {
            uint32_t *tab = tabs.data() + (built % Sh::NB) * Sh::SLOT;
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
            col[buf][t] = column_longest<Sh>(tabs.data(), q, r, w16, m, Ee,
                                             at + t);
        chain_follow<Sh>(chain, col[buf ^ 1].data(), c0, nt, tabs.data(), q,
                         r, w16, m, E, Ee, 0, 1, true);
        if (tabs.back() != kGuard)
            return -1000;
        if (chain.done == 1)
            return chain.count;
        if (chain.done == kChainMany) {
            chain.done = 0;
            all = true;
            continue;
        }
        if (c0 >= 0)
            steps += chain.count - before - (steps >> 2);
        before = chain.count;
        all = steps < 4 * STEPS;
        c0 = at;
        at = std::max(at + nt, chain.c);
        buf ^= 1;
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

// All rows: by a warp (0), by the CTA of index class which - 1.
int emu_rows(const uint32_t *q, const uint32_t *r, int m, int E, int which)
{
    switch (which) {
    case 0: return all_rows<WarpShape>(q, r, m, E);
    case 1: return all_rows<IndexClass<0>::Rows>(q, r, m, E);
    case 2: return all_rows<IndexClass<1>::Rows>(q, r, m, E);
    case 3: return all_rows<IndexClass<2>::Rows>(q, r, m, E);
    default: return all_rows<RowsShape<131072, 8192, kIndexThreads>>(q, r, m,
                                                                     E);
    }
}

int emu_index_rows(const uint32_t *q, const uint32_t *r, int m, int E, int ic,
                   int calm, int *turns)
{
    switch (ic) {
    case 0: return index_rows<0>(q, r, m, E, calm, turns);
    case 1: return index_rows<1>(q, r, m, E, calm, turns);
    default: return index_rows<2>(q, r, m, E, calm, turns);
    }
}

// Whether a thread of the index leaves column c to all rows.
int emu_column(const uint32_t *q, const uint32_t *r, int m, int E, int c)
{
    using Sh = IndexShape0;
    const int w16 = (m + 15) >> 4, Ee = eff_threshold(m, E);
    std::vector<uint32_t> tabs(Sh::WORDS);
    for (int b = std::max(c - Ee, 0) >> Sh::LOGBS;
         b <= std::min(c + Ee, m - 1) >> Sh::LOGBS; ++b) {
        uint32_t *tab = tabs.data() + (b % Sh::NB) * Sh::SLOT;
        table_clear<Sh>(tab, 0, 1);
        table_count<Sh>(tab, q, w16, m, b, 0, 1);
        (void)table_sum<Sh>(tab, 0, 1);
        table_prefix<Sh>(tab, 0, 0, 1);
        table_scatter<Sh>(tab, q, w16, m, b, 0, 1);
    }
    return column_longest<Sh>(tabs.data(), q, r, w16, m, Ee, c) == kColumnMany;
}

// Whether the serving queue takes a pair.
int emu_long_queued(int m, int E)
{
    const int c = class_of_tuned(m, E, serving_params());
    return c >= 0 && long_queued(c);
}

int emu_handed_over(const uint32_t *q, const uint32_t *r, int m, int E)
{
    return handed_over(q, r, m, E);
}

int emu_first_pair(int b, int grid, int sms)
{
    return first_pair(b, grid, sms);
}

int emu_rows_max_e(int which)
{
    switch (which) {
    case 0: return WarpShape::max_e();
    case 1: return IndexClass<0>::Rows::max_e();
    case 2: return IndexClass<1>::Rows::max_e();
    default: return IndexClass<2>::Rows::max_e();
    }
}

}  // extern "C"
