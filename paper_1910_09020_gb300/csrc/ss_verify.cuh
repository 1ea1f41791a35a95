// ss_verify.cuh -- the accuracy harness: exact edit distance (up to E+1) of
// read/reference pairs on the GPU, to measure the filter's false accept and
// false reject rates the way Section 3.2 does with an aligner as ground truth.
// Batches of one length and threshold run bit-sliced (ed_walk of ss_pm.cuh),
// everything else by the diagonals below.
#pragma once
#include <cstdint>

#include "ss_device.cuh"

namespace ssk {

// ---- furthest-reaching diagonals --------------------------------------------
//
// min(ED, E+1) by diagonals instead of table cells (Ukkonen 1985; Landau and
// Vishkin 1989): F_e[k] is the furthest read position i for which the cell
// (i, i + k) costs at most e edits, and
//     F_e[k] = slide(max(F_{e-1}[k] + 1, F_{e-1}[k-1], F_{e-1}[k+1] + 1), k)
// (substitution, reference base inserted, read base dropped), slide running
// along the diagonal while the bases match.  ED is the first e with F_e[0] =
// m.  A path of at most E edits that stands on diagonal k after e of them
// still needs |k| to come back, so only |k| <= min(e, E - e) is kept: about
// E^2 / 2 slides per pair, where the banded table has m (2E+1) cells (10 kbp
// at E = 500: 125 thousand against 10 million).
constexpr int kEdNone = -(1 << 20);  // no cell of this diagonal reached

// Matching bases from q[i], r[j] on, at most n (i + n and j + n inside the
// sequences of w16 packed words).  Two packed words hold the code bits of
// 32 bases from a word's start: 17 to 32 of them are compared at once.
SS_HD int ed_slide(const uint32_t *q, const uint32_t *r, int w16, int i,
                   int j, int n)
{
    int done = 0;
    while (done < n) {
        const int a = i + done, b = j + done;
        const int ia = a >> 4, ib = b >> 4;
        const uint32_t q0 = ldg(q + ia), r0 = ldg(r + ib);
        const uint32_t q1 = ia + 1 < w16 ? ldg(q + ia + 1) : 0u;
        const uint32_t r1 = ib + 1 < w16 ? ldg(r + ib + 1) : 0u;
        const int sa = a & 15, sb = b & 15;
        const uint32_t x =
            ((prmt(q0, q1, 0x5410u) >> sa) ^ (prmt(r0, r1, 0x5410u) >> sb)) |
            ((prmt(q0, q1, 0x7632u) >> sa) ^ (prmt(r0, r1, 0x7632u) >> sb));
        const int valid = 32 - imax(sa, sb);  // bases both windows hold
        const int run = imin(x ? ffs32(x) - 1 : 32, valid);
        done += run;
        if (run < valid)
            break;
    }
    return imin(done, n);
}

// One diagonal: prev points at F_{e-1}[k].
SS_HD int ed_diagonal(const uint32_t *q, const uint32_t *r, int w16, int m,
                      const int *prev, int k)
{
    const int lim = m - imax(k, 0);  // the diagonal's last read position
    int t = imax(imax(prev[0], prev[1]) + 1, prev[-1]);
    t = imin(t, lim);
    return t + ed_slide(q, r, w16, t, t + k, lim - t);
}

// Whether edit count e is the pair's last one: its distance in ed then
// (at = F_e[0]).
SS_HD bool ed_ends(int at, int m, int E, int e, int &ed)
{
    const bool there = at >= m;
    ed = there ? e : E + 1;
    return there || e == E;
}

// F_{e+1} (next) from F_e (prev, both at diagonal 0; e < E), by lane t of a
// team of nt; what lies outside |k| <= min(e, E - e) of prev is kEdNone or
// an older value, which is no further.
SS_HD void ed_advance(const uint32_t *q, const uint32_t *r, int w16, int m,
                      int E, int e, const int *prev, int *next, int t, int nt)
{
    const int w = imin(e + 1, E - e - 1);
    for (int k = t - w; k <= w; k += nt)
        next[k] = ed_diagonal(q, r, w16, m, prev + k, k);
}

// min(ED, E+1) of one pair, its diagonals one after another.
template <int E>
SS_HD int ed_banded(const uint32_t *q, const uint32_t *r, int m, int w16)
{
    constexpr int H = E / 2;
    int F[2][2 * H + 3];
    for (int x = 0; x < 2 * H + 3; ++x)
        F[0][x] = F[1][x] = kEdNone;
    F[0][H + 1] = ed_slide(q, r, w16, 0, 0, m);
    for (int e = 0; e <= E; ++e) {
        const int *prev = F[e & 1] + H + 1;
        if (prev[0] >= m)
            return e;
        const int w = imin(e + 1, E - e - 1);
        for (int k = -w; k <= w; ++k)
            F[(e + 1) & 1][H + 1 + k] =
                ed_diagonal(q, r, w16, m, prev + k, k);
    }
    return E + 1;
}

}  // namespace ssk
