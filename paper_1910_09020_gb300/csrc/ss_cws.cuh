// ss_cws.cuh -- K4 for thresholds from 32 to 816: a team of two or four lanes
// per pair over a window of the sequences.
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

// Code bits of the 17 to 32 bases a sequence's words hold from base j on
// (the number in n): bit t of lo/hi is base j + t.
SS_HD void base_window(const uint32_t *g, int w16, int j, uint32_t &lo,
                       uint32_t &hi, int &n)
{
    const int i = j >> 4, s = j & 15;
    const uint32_t a = ldg(g + i), b = i + 1 < w16 ? ldg(g + i + 1) : 0u;
    lo = prmt(a, b, 0x5410u) >> s;
    hi = prmt(a, b, 0x7632u) >> s;
    n = 32 - s;
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

// Shape of a ring class: rings of QB bases of the query and RB of the
// reference, filled in blocks of BP; LANES lanes per pair.
constexpr int kRingAhead = 159;  // columns read past c (and past c + E)
template <int QB_, int RB_, int BP_, int LANES_ = 4>
struct RingShape {
    static constexpr int QB = QB_, RB = RB_, BP = BP_, LANES = LANES_;
    static constexpr int QW = QB / 32, RW = RB / 32;
    // words of a pair: both rings as (low, high) code words of 32 bases, the
    // first again after the last
    static constexpr int WORDS = 2 * (QW + 1 + RW + 1);
    // the window, what is read past it and the block being filled
    static constexpr int max_e() { return (QB - BP - kRingAhead - 1) / 2; }
    // words a lane goes through in a step: 2E + 1 starts touch at most
    // (2E + 31) / 32 + 1
    static constexpr int LW =
        ((2 * max_e() + 31) / 32 + 1 + LANES - 1) / LANES;
    static_assert(32 % LANES == 0 && BP / 32 % LANES == 0,
                  "a team's lanes fill a block");
    static_assert(LW <= 32, "a lane's words in a mask");
    static_assert(RB >= BP + kRingAhead + 1, "a step in the reference's ring");
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
        const uint32_t a = 2 * i < w16 ? ldg(g + 2 * i) : 0u;
        const uint32_t b = 2 * i + 1 < w16 ? ldg(g + 2 * i + 1) : 0u;
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

// Most columns that a start of the words of lane tl matches, of those that
// match four (0: none does; below four: the query ends there).  open: a
// start that matches 32 and has more, else -1.  keep: the lane's scratch,
// Sh::LW words `stride` apart.
template <class Sh>
SS_HD int ring_lane(const RingStep &s, int tl, uint32_t *keep, int stride,
                    int &open)
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
                run = ring_far(s, j, 32, lim);
        }
        best = imax(best, run);
    }
    return best;
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

#ifdef __CUDACC__
constexpr int kRingWarps = 2;  // warps per CTA

// Shared words of a CTA: its pairs' rings and its lanes' scratch.
template <class Sh>
constexpr size_t ring_smem_words()
{
    return (size_t)kRingWarps * (32 / Sh::LANES * Sh::WORDS + 32 * Sh::LW);
}

template <class Sh>
__global__ void __launch_bounds__(32 * kRingWarps) k_cw_ring(const CwArgs a)
{
    extern __shared__ uint2 rings[];
    constexpr int LANES = Sh::LANES, PAIRS = 32 / LANES;
    const int lane = threadIdx.x & 31, tl = lane % LANES, team = lane / LANES;
    uint2 *q2 = rings + (size_t)((threadIdx.x >> 5) * PAIRS + team) *
                            (Sh::WORDS / 2);
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
    bool alive = false, more = true;
    int64_t p = 0;
    int E = 0, Ee = 0, count = 0;
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
                    count = 0;
                    qn = rn = 0;
                    alive = true;
                } else {
                    more = false;
                }
                s.c = 0;
            }
        }
        if (!__any_sync(0xffffffffu, alive))
            break;
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
            int best = ring_lane<Sh>(s, tl, keep, 32 * kRingWarps,
                                     open);
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
                if (rows != 0u) {
                    const int lim = s.m - max(j, s.c);
                    if (ends == 0u && all < lim)
                        all = ring_far(s, j, all, lim);
                    best = max(best, all);
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
                stop = over || s.c >= until;
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
