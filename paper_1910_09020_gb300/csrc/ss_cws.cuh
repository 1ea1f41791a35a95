// ss_cws.cuh -- K4 for thresholds from 32 to 816: a team of two or four lanes
// per pair over a window of the sequences, or (few pairs, and pairs whose
// rows mostly match, as in a repeat) a warp per pair.
//
// Method (Section 2.4): from checkpoint c the longest escape segment is the
// longest match of R[c..] with the query from any start j in c-E..c+E (row
// s = j - c).
//   1. The starts are taken 32 to a word (starts 32i..32i+31), a word per
//      lane in turn: those that match four bases come from six funnel shifts
//      and eight logic operations on the query's two code planes, and go to
//      the lane's scratch.
//   2. The few survivors (one by chance per 8 words, and the true row's) are
//      compared over 32 columns, those of all lanes side by side; the starts
//      below and above the window are dropped here, not word by word.
//   3. A row that matches all 32 is followed by the whole team, 32 columns
//      per lane at a time; a second one of the same lane by that lane.
//   4. The farthest first obstacle over the team is the next checkpoint.  If
//      no start matches four bases (or the query ends before), the team goes
//      through all words again for the longest prefix.
//
// Bound by instruction issue.  What a step costs besides its words (windows
// of R, survivors, the team's maximum, the chain) is shared by the 8 or 16
// pairs of a warp, which step together, so more words per lane are cheaper
// than more lanes.  2M pairs of 64 bp to 10 kbp at E = 5 %, by E' in ms, one
// word per lane (8, 16 or 32 lanes a pair, the whole pair staged) -> here:
// to 112 2.2 -> 1.3, to 304 about 8 -> 4.2, to 500 about 10 -> 5.5; the
// batch 21.6 -> 11.6.  Other widths: four lanes to 112 1.55; two to 304 4.3
// and to 500 6.7; eight to 500 6.1.  48 registers instead of 64 (20 CTAs per
// SM instead of 16): 1.45, 4.5, 5.8.
//
// The planes are rings, filled up to their end whenever a team of the warp
// gets to the end of its own: all teams then fill theirs together, each with
// its own lanes, so a warp stops for memory once in some 25 steps, and a
// pair takes 0.3 to 0.8 KB of shared memory whatever its length.
#pragma once
#include <cstdint>

#include "ss_bucket.cuh"
#include "ss_cw.cuh"
#include "ss_device.cuh"

namespace ssk {

// A packed word of a sequence, by an ordinary load: the serving queue's worker
// runs these routes while other kernels write the sequences of later pairs,
// and the read-only path (ldg) is for memory that no one writes during the
// kernel.
SS_HD uint32_t seq_word(const uint32_t *p) { return *p; }

// Code bits of the 17 to 32 bases a sequence's words hold from base j on
// (the number in n): bit t of lo/hi is base j + t.
SS_HD void base_window(const uint32_t *g, int w16, int j, uint32_t &lo,
                       uint32_t &hi, int &n)
{
    const int i = j >> 4, s = j & 15;
    const uint32_t a = seq_word(g + i), b = i + 1 < w16 ? seq_word(g + i + 1) : 0u;
    lo = prmt(a, b, 0x5410u) >> s;
    hi = prmt(a, b, 0x7632u) >> s;
    n = 32 - s;
}

// Code bits of bases j..j+31 (those past the last word: 0).
SS_HD void full_window(const uint32_t *g, int w16, int j, uint32_t &lo,
                       uint32_t &hi)
{
    const int i = j >> 4;
    const uint32_t a = seq_word(g + i), b = i + 1 < w16 ? seq_word(g + i + 1) : 0u;
    const uint32_t z = i + 2 < w16 ? seq_word(g + i + 2) : 0u;
    lo = funnel_r(prmt(a, b, 0x5410u), z & 0xffffu, (uint32_t)j & 15u);
    hi = funnel_r(prmt(a, b, 0x7632u), z >> 16, (uint32_t)j & 15u);
}

// Matching bases of q[j..] and r[c..], at most lim (inside both), over at
// most `windows` windows (0: any number): kRunOpen + the bases compared if
// all of them match and more are left.  rlo, rhi, rn: the window of r at c.
constexpr int kRunOpen = 1 << 24;
SS_HD int index_run(const uint32_t *q, const uint32_t *r, int w16, int j,
                    int c, int lim, uint32_t rlo, uint32_t rhi, int rn,
                    int windows)
{
    int run = 0;
    for (;;) {
        uint32_t lo, hi;
        int n;
        base_window(q, w16, j + run, lo, hi, n);
        n = imin(n, rn);
        const uint32_t x = (lo ^ rlo) | (hi ^ rhi);
        const int k = imin(x ? ffs32(x) - 1 : 32, n);
        run += k;
        if (k < n || run >= lim)
            return imin(run, lim);
        if (--windows == 0)
            return run + kRunOpen;
        base_window(r, w16, c + run, rlo, rhi, rn);
    }
}

// Columns read past c (and past c + E) by a team of up to four lanes; a warp
// reads 32 per lane after the first 32.
constexpr int kRingAhead = 159;
// Shape of a ring class: rings of QB bases of the query and RB of the
// reference, filled in blocks of BP; LANES lanes per pair; CTAS of its
// kernel on an SM (14: 72 registers, 12: 80.  Of the largest class, E' = 750,
// 30,000 pairs of 10 kbp 3.07 -> 2.64 ms with 12, 8,000 as much; of the others
// 2M pairs of 64 bp to 10 kbp at 5 % 11.6 -> 11.8).
template <int QB_, int RB_, int BP_, int LANES_ = 4, int CTAS_ = 14>
struct RingShape {
    static constexpr int QB = QB_, RB = RB_, BP = BP_, LANES = LANES_;
    static constexpr int CTAS = CTAS_;
    static constexpr int QW = QB / 32, RW = RB / 32;
    static constexpr int AHEAD = LANES <= 4 ? kRingAhead : 32 * LANES + 95;
    // words of a pair: both rings as (low, high) code words of 32 bases, the
    // first again after the last
    static constexpr int WORDS = 2 * (QW + 1 + RW + 1);
    // the window, what is read past it and the block being filled
    static constexpr int max_e() { return (QB - BP - AHEAD - 1) / 2; }
    // words a lane goes through in a step: 2E + 1 starts touch at most
    // (2E + 31) / 32 + 1
    static constexpr int LW =
        ((2 * max_e() + 31) / 32 + 1 + LANES - 1) / LANES;
    static_assert(32 % LANES == 0 && BP / 32 % LANES == 0,
                  "a team's lanes fill a block");
    static_assert(LW <= 32, "a lane's words in a mask");
    static_assert(RB >= BP + AHEAD + 1, "a step in the reference's ring");
};

// Code bits of bases j..j+31 of a ring of W words.
template <int W>
SS_HD void ring_window(const uint2 *x, int j, uint32_t &lo, uint32_t &hi)
{
    const uint2 *p = x + ((j >> 5) & (W - 1));
    const uint2 a = p[0], b = p[1];
    lo = funnel_r(a.x, b.x, (uint32_t)j & 31u);
    hi = funnel_r(a.y, b.y, (uint32_t)j & 31u);
}

// Load the block from base n on of a sequence into its ring (lane t of nt).
template <int W, int BP>
SS_HD void ring_load(uint2 *x, const uint32_t *g, int w16, int n, int t,
                     int nt)
{
#pragma unroll
    for (int k = 0; k < BP / 32; k += nt) {
        const int i = (n >> 5) + k + t, at = i & (W - 1);
        const uint32_t a = 2 * i < w16 ? seq_word(g + 2 * i) : 0u;
        const uint32_t b = 2 * i + 1 < w16 ? seq_word(g + 2 * i + 1) : 0u;
        const uint2 v =
            make_uint2(prmt(a, b, 0x5410u), prmt(a, b, 0x7632u));
        x[at] = v;
        if (at == 0)
            x[W] = v;
    }
}

// The same from base n0 to base n1 (multiples of 32; lane t of nt).
template <int W>
SS_HD void ring_fill(uint2 *x, const uint32_t *g, int w16, int n0, int n1,
                     int t, int nt)
{
    for (int i = (n0 >> 5) + t; i < n1 >> 5; i += nt) {
        const int at = i & (W - 1);
        const uint32_t a = 2 * i < w16 ? seq_word(g + 2 * i) : 0u;
        const uint32_t b = 2 * i + 1 < w16 ? seq_word(g + 2 * i + 1) : 0u;
        const uint2 v =
            make_uint2(prmt(a, b, 0x5410u), prmt(a, b, 0x7632u));
        x[at] = v;
        if (at == 0)
            x[W] = v;
    }
}

// Whether the block from base n on may be filled (it overwrites bases before
// the window's first) and the column from which a step needs it; first: the
// window's first base, ahead: the last base read past c.
SS_HD bool ring_room(int n, int m, int first, int ring, int bp)
{
    return n < m && n + bp - ring <= imax(first, 0);
}
SS_HD int ring_until(int n, int m, int ahead)
{
    return n < m ? n - ahead : m;
}

// What a step looks at, the same for the lanes of a team.
struct RingStep {
    const uint2 *q2, *r2;    // the rings
    const uint32_t *q, *r;   // packed sequences
    int w16, m, c, lo, hi;
    uint32_t rlo, rhi;       // code bits of R[c..c+31]
};

// Columns that the row starting at j matches from column c + at on, from
// global memory; lim: its columns in all.
SS_HD int ring_far(const RingStep &s, int j, int at, int lim)
{
    uint32_t rlo, rhi;
    int rn;
    base_window(s.r, s.w16, s.c + at, rlo, rhi, rn);
    return at + index_run(s.q, s.r, s.w16, j + at, s.c + at, lim - at, rlo,
                          rhi, rn, 0);
}

// The run of the row starting at j from column c, at most lim bases: every
// lane of a warp calls it (on the host, one lane does all).
SS_HD int warp_run(const uint32_t *q, const uint32_t *r, int w16, int j,
                   int c, int lim)
{
#ifdef __CUDA_ARCH__
    const int lane = threadIdx.x & 31;
    for (int at = 0;; at += 32 * 16) {
        const int o = at + 16 * lane;
        int k = 0;
        if (o < lim) {
            uint32_t qlo, qhi, rlo, rhi;
            int qn, rn;
            base_window(q, w16, j + o, qlo, qhi, qn);
            base_window(r, w16, c + o, rlo, rhi, rn);
            const uint32_t x = (qlo ^ rlo) | (qhi ^ rhi);
            k = imin(x ? ffs32(x) - 1 : 16, 16);
        }
        const uint32_t stop = __ballot_sync(0xffffffffu, k < 16);
        if (stop) {
            const int f = __ffs((int)stop) - 1;
            return imin(__shfl_sync(0xffffffffu, o + k, f), lim);
        }
    }
#else
    uint32_t rlo, rhi;
    int rn;
    base_window(r, w16, c, rlo, rhi, rn);
    return index_run(q, r, w16, j, c, lim, rlo, rhi, rn, 0);
#endif
}

// Columns of R[c + at .. c + at + 31] that the row starting at j matches
// (negative: it ends before).
template <class Sh>
SS_HD int ring_match(const RingStep &s, int j, int at)
{
    uint32_t ql, qh, rl, rh;
    ring_window<Sh::QW>(s.q2, j + at, ql, qh);
    ring_window<Sh::RW>(s.r2, s.c + at, rl, rh);
    const uint32_t x = (ql ^ rl) | (qh ^ rh);
    return imin(x ? ffs32(x) - 1 : 32, s.m - imax(j, s.c) - at);
}

// The same from column c + at on, as far as the rings reach and then from
// global memory; lim: the row's columns in all, at < lim.
template <class Sh>
SS_HD int ring_follow(const RingStep &s, int j, int at, int lim)
{
    for (; at + 31 <= Sh::AHEAD && at < lim; at += 32) {
        const int run = ring_match<Sh>(s, j, at);
        if (run < 32)
            return at + run;
    }
    return at < lim ? ring_far(s, j, at, lim) : lim;
}

// Most columns that a start of the words of lane tl matches, of those that
// match four (0: none does; below four: the query ends there).  open: a
// start that matches 32 and has more, else -1.  keep: the lane's scratch,
// Sh::LW words `stride` apart.  work: grows by the comparisons of 32 columns
// that the survivors took.
template <class Sh>
SS_HD int ring_lane(const RingStep &s, int tl, uint32_t *keep, int stride,
                    int &open, int &work)
{
    uint32_t pl[4], ph[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        pl[k] = 0u - ((s.rlo >> k) & 1u);
        ph[k] = 0u - ((s.rhi >> k) & 1u);
    }
    // the survivors of all words first, so that the lanes of a warp then
    // compare theirs side by side
    const int i0 = (s.lo >> 5) + tl;
    uint32_t hits = 0u, bit = 1u, *kp = keep;
    for (int i = i0; i <= s.hi >> 5; i += Sh::LANES) {
        const uint2 *p = s.q2 + (i & (Sh::QW - 1));
        const uint2 a = p[0], b = p[1];
        uint32_t y = (a.x ^ pl[0]) | (a.y ^ ph[0]);
#pragma unroll
        for (int k = 1; k < 4; ++k) {
            y |= funnel_r(a.x, b.x, k) ^ pl[k];
            y |= funnel_r(a.y, b.y, k) ^ ph[k];
        }
        *kp = ~y;
        hits |= ~y ? bit : 0u;
        kp += stride;
        bit += bit;
    }
    int best = 0, i = 0;
    uint32_t S = 0u;
    open = -1;
    while (hits | S) {
        if (S == 0u) {
            const int k = ffs32(hits) - 1;
            hits &= hits - 1u;
            S = keep[k * stride];
            i = i0 + Sh::LANES * k;
        }
        const int t = ffs32(S) - 1, j = 32 * i + t;
        S &= S - 1u;
        ++work;
        const uint2 *p = s.q2 + (i & (Sh::QW - 1));
        const uint2 a = p[0], b = p[1];
        const uint32_t x = (funnel_r(a.x, b.x, (uint32_t)t) ^ s.rlo) |
                           (funnel_r(a.y, b.y, (uint32_t)t) ^ s.rhi);
        const int lim = s.m - imax(j, s.c);  // query or row end
        int run = imin(x ? ffs32(x) - 1 : 32, lim);
        if ((uint32_t)(j - s.lo) > (uint32_t)(s.hi - s.lo))
            run = 0;  // outside the window
        if (run == 32 && lim > 32) {
            if (open < 0)
                open = j;
            else
                run = ring_follow<Sh>(s, j, 32, lim);
            work += run >> 5;
        }
        best = imax(best, run);
    }
    return best;
}
template <class Sh>
SS_HD int ring_lane(const RingStep &s, int tl, uint32_t *keep, int stride,
                    int &open)
{
    int work = 0;
    return ring_lane<Sh>(s, tl, keep, stride, open, work);
}

// Columns that some start of word i in lo..hi matches from c on, where none
// matches four (or cols < 4 are left): 0..min(3, cols).
template <class Sh>
SS_HD int prefix_word(const RingStep &s, int cols, int i)
{
    const uint2 *p = s.q2 + (i & (Sh::QW - 1));
    const uint2 a = p[0], b = p[1];
    uint32_t y = 0u;
    int best = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        y |= funnel_r(a.x, b.x, k) ^ (0u - ((s.rlo >> k) & 1u));
        y |= funnel_r(a.y, b.y, k) ^ (0u - ((s.rhi >> k) & 1u));
        // starts in the window with k + 1 bases
        const uint32_t range =
            mask_below(imin(s.hi + 1, s.m - k) - 32 * i) &
            ~mask_below(s.lo - 32 * i);
        if (k < cols && (~y & range) != 0u)
            best = k + 1;
    }
    return best;
}

// ---- one pair to a warp or a CTA ----------------------------------------------
//
// What counts here is the time of a step: with few pairs nothing else hides
// it, and a warp alone issues an instruction every three cycles.  A lane takes
// 32 rows, from the window's first start on, so that a warp does with one turn
// up to E' = 511; the columns are gone through until the rows of the whole
// warp are dead, and what is left after eight is nearly always the one true
// row, which all lanes then follow, 32 columns each.

// Votes and shuffles of a warp; on the host a warp is one lane.
SS_HD bool warp_any(bool v)
{
#ifdef __CUDA_ARCH__
    return __any_sync(0xffffffffu, v);
#else
    return v;
#endif
}
SS_HD uint32_t warp_ballot(bool v)
{
#ifdef __CUDA_ARCH__
    return __ballot_sync(0xffffffffu, v);
#else
    return v ? 1u : 0u;
#endif
}
SS_HD int warp_shfl(int v, int lane)
{
#ifdef __CUDA_ARCH__
    return __shfl_sync(0xffffffffu, v, lane);
#else
    (void)lane;
    return v;
#endif
}
SS_HD int popc32(uint32_t x)
{
#ifdef __CUDA_ARCH__
    return __popc(x);
#else
    return __builtin_popcount(x);
#endif
}
SS_HD int warp_max(int v)
{
#ifdef __CUDA_ARCH__
    return __reduce_max_sync(0xffffffffu, v);
#else
    return v;
#endif
}

// Columns that the row starting at j matches from c on, followed by all
// lanes of a warp from column `at` on, 32 columns each and then from global
// memory (j, at and lim, the row's columns, the same for all).
template <class Sh>
SS_HD int warp_follow(const RingStep &s, int j, int at, int lim)
{
#ifdef __CUDA_ARCH__
    if (at + 32 * 31 + 31 > Sh::AHEAD)
        return at + warp_run(s.q, s.r, s.w16, j + at, s.c + at, lim - at);
    const int run = ring_match<Sh>(s, j, at + 32 * (threadIdx.x & 31));
    const unsigned ends = __ballot_sync(0xffffffffu, run < 32);
    const int k = ends ? __ffs((int)ends) - 1 : 31;
    at += 32 * k + __shfl_sync(0xffffffffu, run, k);
    if (ends || at >= lim)
        return imin(at, lim);
    return at + warp_run(s.q, s.r, s.w16, j + at, s.c + at, lim - at);
#else
    return ring_follow<Sh>(s, j, at, lim);
#endif
}

// Code bits of 64 bases.
struct RowWindow {
    uint32_t al, ah, bl, bh;  // the first 32 and the last
};
// Bit t: base t + k of the window is not the base whose code bits fill lo, hi.
SS_HD uint32_t rows_miss(const RowWindow &w, uint32_t lo, uint32_t hi, int k)
{
    return (funnel_r(w.al, w.bl, (uint32_t)k) ^ lo) |
           (funnel_r(w.ah, w.bh, (uint32_t)k) ^ hi);
}
SS_HD uint32_t fill_bit(uint32_t x, int k) { return 0u - ((x >> k) & 1u); }

// Bits 0..3 of x, each filling a word.
SS_HD void fill_bits(uint32_t x, uint32_t (&f)[4])
{
#ifdef __CUDA_ARCH__
    // bit k to the sign of byte k (no two partial products meet), which a
    // byte permutation spreads
    const uint32_t y = (x & 15u) * 0x10204080u;
    asm("prmt.b32 %0, %1, 0, 0x8888;" : "=r"(f[0]) : "r"(y));
    asm("prmt.b32 %0, %1, 0, 0x9999;" : "=r"(f[1]) : "r"(y));
    asm("prmt.b32 %0, %1, 0, 0xaaaa;" : "=r"(f[2]) : "r"(y));
    asm("prmt.b32 %0, %1, 0, 0xbbbb;" : "=r"(f[3]) : "r"(y));
#else
    for (int k = 0; k < 4; ++k)
        f[k] = fill_bit(x, k);
#endif
}

// A lane's survivors (starts j0 + t, bit t of S, that match eight bases, w
// their window) where there are many, as in a repeat: taken on together, four
// columns at a time, until one is left or their row ends.
// Returns the starts left, which match `from` columns; best: the columns
// matched by those that are not.
constexpr int kRingDense = 4;
template <class Sh>
SS_HD uint32_t ring_dense(const RingStep &s, RowWindow w, int j0, uint32_t S,
                          int &best, int &from)
{
    uint32_t rlo = s.rlo, rhi = s.rhi;
    // the window's 64 bases and the reference's 32 exist
    if (j0 + 64 > s.m || s.c + 32 > s.m)
        return S;
    for (int at = 0, d = 8;; d = 0) {
        from = at;
        for (; d < 32; d += 4) {
            uint32_t lo[4], hi[4], on = S;
            fill_bits(rlo >> d, lo);
            fill_bits(rhi >> d, hi);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                on &= ~rows_miss(w, lo[k], hi[k], d + k);
            if (on == 0u) {
                for (int k = 0;; ++k) {
                    S &= ~rows_miss(w, fill_bit(rlo, d + k),
                                    fill_bit(rhi, d + k), d + k);
                    if (S == 0u) {
                        best = imax(best, at + d + k);
                        return 0u;
                    }
                }
            }
            S = on;
            if ((S & (S - 1u)) == 0u)
                return S;
        }
        from = at += 32;
        if (j0 + at + 64 > s.m || s.c + at + 32 > s.m)
            return S;
        w.al = w.bl;
        w.ah = w.bh;
        if (at + 63 <= Sh::AHEAD) {
            ring_window<Sh::QW>(s.q2, j0 + at + 32, w.bl, w.bh);
            ring_window<Sh::RW>(s.r2, s.c + at, rlo, rhi);
        } else {
            full_window(s.q, s.w16, j0 + at + 32, w.bl, w.bh);
            full_window(s.r, s.w16, s.c + at, rlo, rhi);
        }
    }
}

// Longest run of a lane's survivors, which match `from` columns, each by
// itself; open: the first (if it is the only one, or they were not taken on
// together) that matches 32 and has more, else -1.
template <class Sh>
SS_HD int ring_single(const RingStep &s, const RowWindow &w, int j0,
                      uint32_t S, int from, int best, int &open)
{
    const bool one = from == 0 || (S & (S - 1u)) == 0u;
    for (; S; S &= S - 1u) {
        const uint32_t t = (uint32_t)(ffs32(S) - 1);
        const int j = j0 + (int)t;
        const int lim = s.m - imax(j, s.c);  // query or row end
        if (lim <= best)
            continue;
        const uint32_t x = (funnel_r(w.al, w.bl, t) ^ s.rlo) |
                           (funnel_r(w.ah, w.bh, t) ^ s.rhi);
        int run = imin(x ? ffs32(x) - 1 : 32, lim);
        if (run == 32 && lim > 32) {
            if (open < 0 && one)
                open = j;
            else
                run = ring_follow<Sh>(s, j, imax(from, 32), lim);
        }
        best = imax(best, run);
    }
    return best;
}

// The starts of S that still match after columns A to B - 1 (ENDS: the
// query's or the row's end may come first).  False: none does, in no lane.
template <bool ENDS, int A, int B, int NW>
SS_HD bool rows_columns(const RingStep &s, const RowWindow (&w)[NW],
                        const uint32_t (&lo)[4], const uint32_t (&hi)[4],
                        int j0, int stride, uint32_t (&S)[NW])
{
    uint32_t any = 0u;
#pragma unroll
    for (int n = 0; n < NW; ++n) {
#pragma unroll
        for (int k = A; k < B; ++k) {
            S[n] &= ~rows_miss(w[n], lo[k & 3], hi[k & 3], k);
            if (ENDS)
                S[n] = s.c + k < s.m
                           ? S[n] & mask_below(s.m - k - j0 - n * stride)
                           : 0u;
        }
        any |= S[n];
    }
    return warp_any(any != 0u);
}

// Longest run, of four columns or more (else 0), of the rows of the warp's
// lanes in the window: lane t of the team takes the starts lo + 32 t + k
// stride..., NW words of 32 at a time.  many: set where a lane had many
// survivors.  The result is the same in every lane.
template <class Sh, bool ENDS, int NW>
SS_HD int rows_step(const RingStep &s, int t, int stride, bool &many)
{
    int best = 0;
    for (int j0 = s.lo + 32 * t; warp_any(j0 <= s.hi); j0 += NW * stride) {
        RowWindow w[NW];
        uint32_t S[NW], lo[4], hi[4];
        fill_bits(s.rlo, lo);
        fill_bits(s.rhi, hi);
#pragma unroll
        for (int n = 0; n < NW; ++n) {
            const int j = j0 + n * stride;
            ring_window<Sh::QW>(s.q2, j, w[n].al, w[n].ah);
            ring_window<Sh::QW>(s.q2, j + 32, w[n].bl, w[n].bh);
            S[n] = mask_below(s.hi + 1 - j);
        }
        if (!rows_columns<ENDS, 0, 4>(s, w, lo, hi, j0, stride, S))
            continue;
        best = imax(best, 4);
        fill_bits(s.rlo >> 4, lo);
        fill_bits(s.rhi >> 4, hi);
        if (!rows_columns<ENDS, 4, 5>(s, w, lo, hi, j0, stride, S))
            continue;
        best = imax(best, 5);
        if (!rows_columns<ENDS, 5, 6>(s, w, lo, hi, j0, stride, S))
            continue;
        best = imax(best, 6);
        if (!rows_columns<ENDS, 6, 7>(s, w, lo, hi, j0, stride, S))
            continue;
        best = imax(best, 7);
        if (!rows_columns<ENDS, 7, 8>(s, w, lo, hi, j0, stride, S))
            continue;
        best = imax(best, 8);
        uint32_t left = 0u;  // a lane's survivors, one of them told exactly
        int first = 0;
#pragma unroll
        for (int n = 0; n < NW; ++n) {
            if (S[n])
                first = j0 + n * stride + ffs32(S[n]) - 1;
            left = (left && S[n]) ? 3u : left | S[n];
        }
        uint32_t rows = warp_ballot(left != 0u);
        if ((rows & (rows - 1u)) == 0u &&
            !warp_any((left & (left - 1u)) != 0u)) {
            // one row
            const int j = warp_shfl(first, ffs32(rows) - 1);
            best = imax(best,
                        warp_follow<Sh>(s, j, 8, s.m - imax(j, s.c)));
            continue;
        }
        int own = best, open = -1;
#pragma unroll
        for (int n = 0; n < NW; ++n) {
            const int j = j0 + n * stride;
            int from = 0;
            if (popc32(S[n]) > kRingDense) {
                many = true;
                S[n] = ring_dense<Sh>(s, w[n], j, S[n], own, from);
            }
            own = ring_single<Sh>(s, w[n], j, S[n], from, own, open);
        }
        rows = warp_ballot(open >= 0);
        int at = 32;
        // several: each by its lane, until few are left or the rings end
        while (popc32(rows) > (at < 96 ? 1 : 4) && at + 31 <= Sh::AHEAD) {
            if (open >= 0) {
                const int run = ring_match<Sh>(s, open, at);
                if (run < 32) {
                    own = imax(own, at + run);
                    open = -1;
                }
            }
            at += 32;
            rows = warp_ballot(open >= 0);
        }
        best = warp_max(own);
        for (; rows; rows &= rows - 1u) {
            const int j = warp_shfl(open, ffs32(rows) - 1);
            best = imax(best,
                        warp_follow<Sh>(s, j, at, s.m - imax(j, s.c)));
        }
    }
    return best;
}
template <class Sh>
SS_HD int rows_step(const RingStep &s, int t, int stride, bool &many)
{
    // the last start's eighth base, and the eighth column; one word each, or
    // two side by side (E' = 800 by a warp, 152 pairs: 305 us, one after the
    // other 407)
    const bool ends = s.hi + 8 > s.m - 1 || s.c + 8 > s.m;
    if (s.hi - s.lo < stride)
        return ends ? rows_step<Sh, true, 1>(s, t, stride, many)
                    : rows_step<Sh, false, 1>(s, t, stride, many);
    return ends ? rows_step<Sh, true, 2>(s, t, stride, many)
                : rows_step<Sh, false, 2>(s, t, stride, many);
}

// A pair of a ring class taken by a warp: whichever class, its rings fit
// where the warp's teams keep theirs.  (With rings of half the size the warp
// of a 100 kbp pair waited for memory a hundred times instead of twenty.)
using WarpShape = RingShape<8192, 8192, 1024, 32>;
static_assert(WarpShape::max_e() >= ring_max_e(kRingClasses - 1),
              "the classes' thresholds fit a warp's rings");

// Comparisons of 32 columns that a lane of a team may spend on the survivors
// of a pair's first c columns and `count` steps before the warp takes the
// pair (random bases: the rows' share of c, and up to 1.6 a step).
SS_HD int ring_work_limit(int c, int count)
{
    return 256 + 4 * count + (c >> 4);
}

// A class of up to this many pairs per two warps of its launch is routed a
// pair at a time by each (c: ring class): side by side they wait for one
// another's steps, 1.3 us each, and too few warps stand on the GPU to hide
// it.  n pairs of 2 kbp at E' = 100, 6 kbp at 290 and 10 kbp at 490, us, side
// by side / a pair to a warp / a warp for each from the start, the whole pair
// staged: n = 4000 309 / 153 / 223, 672 / 334 / 444, 1085 / 515 / 503; n =
// 16000 331 / 394, 820 / 750, 1482 / 1370 against 332, 815, 1282.  When no
// more pairs are waiting, so are a warp's last few.
constexpr int ring_few(int c) { return c < 2 ? 4 : 7; }
constexpr int kRingLast = 2;

#ifdef __CUDACC__
constexpr int kRingWarps = 2;  // warps per CTA

// Shared words of a CTA: its pairs' rings and its lanes' scratch.
template <class Sh>
constexpr size_t ring_smem_words()
{
    static_assert(32 / Sh::LANES * Sh::WORDS >= WarpShape::WORDS,
                  "a warp's rings in its teams'");
    return (size_t)kRingWarps * (32 / Sh::LANES * Sh::WORDS + 32 * Sh::LW);
}

template <class T>
__device__ __forceinline__ const T *shfl_ptr(const T *p, int lane)
{
    return reinterpret_cast<const T *>(
        __shfl_sync(0xffffffffu, (unsigned long long)p, lane));
}

// The pair (of the class's first gridDim.x) that a CTA takes without waiting
// for the counter, sms of them over all SMs.  CTAs come to the SMs in rounds
// of one each if these are free; if other classes' CTAs still leave, the
// first dozens come to the few that are free.  So an SM's pairs (sms apart)
// are dealt to rounds that differ from SM to SM: 129 pairs beside other
// classes stood on 10 SMs in the order of the CTAs, on 115 and more dealt.
SS_HD int first_pair(int b, int grid, int sms)
{
    const int rounds = grid / sms;
    if (rounds < 2 || b >= rounds * sms)
        return b;
    const int x = b % sms, k = (b / sms + 5 * x) % rounds;
    return x + sms * k;
}

// The rest of a pair from checkpoint s.c and `count` obstacles on, by the
// whole warp; x: its rings.  Returns the pair's obstacles, min(count, E+1).
template <class Sh>
__device__ __forceinline__ int warp_route(RingStep s, int E, int Ee,
                                          int count, uint2 *x)
{
    const int lane = threadIdx.x & 31;
    uint2 *r2 = x + Sh::QW + 1;
    s.q2 = x;
    s.r2 = r2;
    int qn = 0, rn = 0;
    for (;;) {
        qn = max(qn, max(s.c - Ee, 0) & ~(Sh::BP - 1));
        rn = max(rn, s.c & ~(Sh::BP - 1));
        for (; ring_room(qn, s.m, s.c - Ee, Sh::QB, Sh::BP); qn += Sh::BP)
            ring_load<Sh::QW, Sh::BP>(x, s.q, s.w16, qn, lane, 32);
        for (; ring_room(rn, s.m, s.c, Sh::RB, Sh::BP); rn += Sh::BP)
            ring_load<Sh::RW, Sh::BP>(r2, s.r, s.w16, rn, lane, 32);
        const int until = min(ring_until(qn, s.m, Ee + Sh::AHEAD),
                              ring_until(rn, s.m, Sh::AHEAD));
        __syncwarp();
        do {
            ring_window<Sh::RW>(r2, s.c, s.rlo, s.rhi);
            s.lo = max(s.c - Ee, 0);
            s.hi = min(s.c + Ee, s.m - 1);
            bool many = false;
            int best = rows_step<Sh>(s, lane, 1024, many);
            if (best < 4) {
                int pre = 0;
                for (int i = (s.lo >> 5) + lane; i <= s.hi >> 5; i += 32)
                    pre = max(pre, prefix_word<Sh>(s, s.m - s.c, i));
                best = __reduce_max_sync(0xffffffffu, pre);
            }
            s.c += best + 1;
            count += s.c <= s.m ? 1 : 0;
            if (s.c >= s.m || count > E)
                return count;
        } while (s.c < until);
        __syncwarp();  // the rings are written again
    }
}

// Columns that the row starting at j matches from c on, followed from column
// `at` on by the lanes of a team, 16 columns each from global memory; on:
// whether the team has a row to follow (every lane of the warp calls it).
template <int LANES>
__device__ __forceinline__ int team_far(const RingStep &s, int j, int at,
                                        int lim, bool on)
{
    const int lane = threadIdx.x & 31, tl = lane % LANES, t0 = lane - tl;
    while (__any_sync(0xffffffffu, on)) {
        int k = 0;
        const int o = at + 16 * tl;
        if (on && o < lim) {
            uint32_t qlo, qhi, rlo, rhi;
            int qn, rn;
            base_window(s.q, s.w16, j + o, qlo, qhi, qn);
            base_window(s.r, s.w16, s.c + o, rlo, rhi, rn);
            const uint32_t y = (qlo ^ rlo) | (qhi ^ rhi);
            k = min(y ? ffs32(y) - 1 : 16, 16);
        }
        const unsigned ends = (__ballot_sync(0xffffffffu, k < 16) >> t0) &
                              ((1u << LANES) - 1u);
        const int f = ends ? __ffs((int)ends) - 1 : LANES - 1;
        k = __shfl_sync(0xffffffffu, k, f, LANES);
        if (on) {
            at += 16 * f + k;
            on = ends == 0u && at < lim;
        }
    }
    return min(at, lim);
}

template <class Sh>
__global__ void __launch_bounds__(32 * kRingWarps, Sh::CTAS)
    k_cw_ring(const CwArgs a)
{
    extern __shared__ uint2 rings[];
    constexpr int LANES = Sh::LANES, PAIRS = 32 / LANES;
    const int lane = threadIdx.x & 31, tl = lane % LANES, team = lane / LANES;
    uint2 *const x =
        rings + (size_t)(threadIdx.x >> 5) * PAIRS * (Sh::WORDS / 2);
    uint2 *q2 = x + team * (Sh::WORDS / 2);
    uint2 *r2 = q2 + Sh::QW + 1;
    uint32_t *keep =
        reinterpret_cast<uint32_t *>(rings + kRingWarps * PAIRS *
                                                 (Sh::WORDS / 2)) +
        threadIdx.x;
    RingStep s;
    s.q2 = q2;
    s.r2 = r2;
    s.q = s.r = nullptr;
    s.w16 = s.m = 1;
    s.c = 0;
    const int begin = a.ws.ranges[2 * a.cls];
    const int end = a.ws.ranges[2 * a.cls + 1];
    const int warps = kRingWarps * (int)gridDim.x;
    // few pairs: one to a warp
    const bool few = 2 * (int64_t)(end - begin) <=
                     (int64_t)ring_few(a.cls - kFirstRing) * warps;
    if (few) {
        // (CTAs stand on two of an SM's four schedulers in turn, a warp on
        // each: the first pairs on one of a CTA's warps, every two the other)
        const int turn = (int)blockIdx.x / (2 * a.sms) & 1;
        int idx = begin + first_pair((int)blockIdx.x, (int)gridDim.x, a.sms) +
                  ((int)(threadIdx.x >> 5) ^ turn) * (int)gridDim.x;
        while (idx < end) {
            const int64_t p = a.ws.perm[idx];
            const int64_t off = a.ps.off(p);
            const int E = a.ps.thr(p);
            s.m = a.ps.len(p);
            s.w16 = (s.m + 15) >> 4;
            s.q = a.ps.reads + off;
            s.r = a.ps.refs + off;
            const int n =
                warp_route<WarpShape>(s, E, eff_threshold(s.m, E), 0, x);
            int next = 0;
            if (lane == 0) {
                a.ps.acc[p] = (uint8_t)(n <= E);
                a.ps.obs[p] = n;
                next = (int)atomicAdd(&a.ws.counters[a.cls], 1u);
            }
            idx = begin + warps + __shfl_sync(0xffffffffu, next, 0);
        }
        return;
    }
    bool alive = false, more = true;
    int64_t p = 0;
    int E = 0, Ee = 0, count = 0, work = 0;
    int qn = 0, rn = 0;  // bases filled in so far
    for (;;) {
        if (__any_sync(0xffffffffu, more && !alive)) {
            int idx = 0;
            if (more && !alive && tl == 0)
                idx = begin + (int)atomicAdd(&a.ws.counters[a.cls], 1u);
            idx = __shfl_sync(0xffffffffu, idx, 0, LANES);
            if (more && !alive) {
                if (idx < end) {
                    p = a.ws.perm[idx];
                    s.m = a.ps.len(p);
                    s.w16 = (s.m + 15) >> 4;
                    E = a.ps.thr(p);
                    Ee = eff_threshold(s.m, E);
                    const int64_t off = a.ps.off(p);
                    s.q = a.ps.reads + off;
                    s.r = a.ps.refs + off;
                    count = work = 0;
                    qn = rn = 0;
                    alive = true;
                } else {
                    more = false;
                }
                s.c = 0;
            }
        }
        // the pairs the whole warp takes: those with too many survivors, and
        // the last few
        const unsigned live = __ballot_sync(0xffffffffu, alive && tl == 0);
        const bool hot =
            (__ballot_sync(0xffffffffu, work > ring_work_limit(s.c, count)) >>
             (team * LANES)) & ((1u << LANES) - 1u);
        unsigned whole = __ballot_sync(
            0xffffffffu, alive && tl == 0 && hot);
        if (__any_sync(0xffffffffu, !more) && __popc(live) <= kRingLast)
            whole = live;
        if (live == 0u)
            break;
        if (whole) {
            for (; whole; whole &= whole - 1u) {
                const int from = __ffs((int)whole) - 1;  // the team's lane 0
                RingStep w;
                w.q = shfl_ptr(s.q, from);
                w.r = shfl_ptr(s.r, from);
                w.w16 = __shfl_sync(0xffffffffu, s.w16, from);
                w.m = __shfl_sync(0xffffffffu, s.m, from);
                w.c = __shfl_sync(0xffffffffu, s.c, from);
                const int n = warp_route<WarpShape>(
                    w, __shfl_sync(0xffffffffu, E, from),
                    __shfl_sync(0xffffffffu, Ee, from),
                    __shfl_sync(0xffffffffu, count, from), x);
                if (team == from / LANES) {
                    if (tl == 0) {
                        a.ps.acc[p] = (uint8_t)(n <= E);
                        a.ps.obs[p] = n;
                    }
                    alive = false;
                    s.c = 0;
                }
                __syncwarp();  // the rings are written again
            }
            qn = rn = 0;  // the others' rings are filled again
            continue;
        }
        // fill the rings; blocks that a long match has passed are left out
        qn = max(qn, max(s.c - Ee, 0) & ~(Sh::BP - 1));
        rn = max(rn, s.c & ~(Sh::BP - 1));
        for (;;) {
            const bool fq =
                alive && ring_room(qn, s.m, s.c - Ee, Sh::QB, Sh::BP);
            const bool fr = alive && ring_room(rn, s.m, s.c, Sh::RB, Sh::BP);
            if (!__any_sync(0xffffffffu, fq || fr))
                break;
            if (fq) {
                ring_load<Sh::QW, Sh::BP>(q2, s.q, s.w16, qn, tl, LANES);
                qn += Sh::BP;
            }
            if (fr) {
                ring_load<Sh::RW, Sh::BP>(r2, s.r, s.w16, rn, tl, LANES);
                rn += Sh::BP;
            }
        }
        const int until = min(ring_until(qn, s.m, Ee + kRingAhead),
                              ring_until(rn, s.m, kRingAhead));
        __syncwarp();
        // step until a team is done with its pair or has to fill its rings
        bool over = false;
        for (;;) {
            ring_window<Sh::RW>(r2, s.c, s.rlo, s.rhi);
            s.lo = max(s.c - Ee, 0);
            s.hi = alive ? min(s.c + Ee, s.m - 1) : -1;
            int open;
            int best = ring_lane<Sh>(s, tl, keep, 32 * kRingWarps, open,
                                     work);
            unsigned rows =
                (__ballot_sync(0xffffffffu, open >= 0) >> (team * LANES)) &
                ((1u << LANES) - 1u);
            while (__any_sync(0xffffffffu, rows != 0u)) {
                const int j = __shfl_sync(0xffffffffu, open,
                                          rows ? __ffs((int)rows) - 1 : 0,
                                          LANES);
                const int at = 32 + 32 * tl;
                const int run = ring_match<Sh>(s, j, at);
                const unsigned ends =
                    (__ballot_sync(0xffffffffu, run < 32) >>
                     (team * LANES)) &
                    ((1u << LANES) - 1u);
                const int k = ends ? __ffs((int)ends) - 1 : LANES - 1;
                int all = 32 + 32 * k + __shfl_sync(0xffffffffu, run, k,
                                                    LANES);
                const int lim = s.m - max(j, s.c);
                const bool on = rows != 0u && ends == 0u && all < lim;
                if (__any_sync(0xffffffffu, on))
                    all = team_far<LANES>(s, j, all, lim, on);
                if (rows != 0u) {
                    best = max(best, min(all, lim));
                    rows &= rows - 1u;
                }
            }
#pragma unroll
            for (int o = LANES / 2; o > 0; o >>= 1)
                best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
            const bool none = alive && best < 4;
            if (__any_sync(0xffffffffu, none)) {
                int pre = 0;
                if (none)
                    for (int i = (s.lo >> 5) + tl; i <= s.hi >> 5; i += LANES)
                        pre = max(pre, prefix_word<Sh>(s, s.m - s.c, i));
#pragma unroll
                for (int o = LANES / 2; o > 0; o >>= 1)
                    pre = max(pre, __shfl_xor_sync(0xffffffffu, pre, o));
                if (none)
                    best = pre;
            }
            // an obstacle at c + best (perhaps on the last column), or the
            // net reached the destination
            bool stop = false;
            if (alive) {
                s.c += best + 1;
                count += s.c <= s.m ? 1 : 0;
                over = s.c >= s.m || count > E;
                stop = over || s.c >= until ||
                       work > ring_work_limit(s.c, count);
            }
            if (__any_sync(0xffffffffu, stop))
                break;
        }
        if (over) {
            if (tl == 0) {
                a.ps.acc[p] = (uint8_t)(count <= E);
                a.ps.obs[p] = count;
            }
            alive = false;
            s.c = 0;
        }
        __syncwarp();  // the rings are written again
    }
}
#endif

}  // namespace ssk
