// ss_cwt.cuh -- K4 for thresholds from 32 to 496: a team of 8, 16 or 32
// lanes per pair, one lane per 32 consecutive query positions.
//
// Method (Section 2.4): from checkpoint c the longest escape segment is the
// longest match of R[c..] with the query from any start j in c-E..c+E (row
// s = j - c).  A lane owns the aligned 32-bit word i of start positions
// 32i..32i+31, so the window of a query plane that column c + d reads for
// all of them is two words funnel-shifted by the constant d.
//   1. Four columns at once, 32 starts per word operation, no branch:
//      S = AND over d = 0..3 of (plane of base R[c+d])[32i + d ..], with one
//      plane per base (bit j of plane b: Q[j] == b, zero outside the query,
//      so Eq. 1 case 4 needs no test).  A random start survives with
//      probability 1/256.
//   2. Each survivor is extended 16 bases per comparison along its row
//      (2-bit codes of query and reference, one funnel shift each).
//   3. The farthest first obstacle over the team is the next checkpoint;
//      without a survivor it lies where the last nonempty prefix of the AND
//      ended.
// Bound by instruction issue (167 per step and warp at E' = 241-307), so what matters
// is that the lanes are busy: the team is the smallest width that covers
// the pair's 2E+1 starts in one word per lane, the teams of a warp step
// together, each on its own pair, and a team that finishes takes its next
// pair while the others keep theirs.  Against one warp per pair evaluating
// column after column with an early exit (216 instructions per step, half
// of the lanes without rows), 2M pairs of 64 bp to 10 kbp at E = 5 %: 32.1
// -> 21.6 ms.
#pragma once
#include <cstdint>

#include "ss_bucket.cuh"
#include "ss_cw.cuh"
#include "ss_device.cuh"

namespace ssk {

// Shared memory of one staged pair: four base planes of PW words (the last
// word zero), then the 2-bit codes of query and reference, QW words each
// (16 bases per word, the words past the end zero; two past it, since a
// window pair from the last base reads them).
struct TeamLayout {
    int PW, QW;
    __host__ __device__ static TeamLayout of(int m)
    {
        const int W32 = (m + 31) >> 5;
        return TeamLayout{W32 + 1, 2 * W32 + 2};
    }
    __host__ __device__ int words() const { return 4 * PW + 2 * QW; }
};

// A packed word (code bit 0 of base t at bit t, code bit 1 at bit 16 + t)
// with the two bits of each base side by side: base t at bits 2t, 2t + 1
// (the outer perfect shuffle).
SS_HD uint32_t interleave_codes(uint32_t x)
{
    uint32_t t = (x ^ (x >> 8)) & 0x0000ff00u;
    x ^= t ^ (t << 8);
    t = (x ^ (x >> 4)) & 0x00f000f0u;
    x ^= t ^ (t << 4);
    t = (x ^ (x >> 2)) & 0x0c0c0c0cu;
    x ^= t ^ (t << 2);
    t = (x ^ (x >> 1)) & 0x22222222u;
    return x ^ t ^ (t << 1);
}

// Stage pair (gq, gr, m) into sm with threads t, t + nt, ...
SS_HD void team_stage(uint32_t *sm, const TeamLayout &L, const uint32_t *gq,
                      const uint32_t *gr, int m, int t, int nt)
{
    const int W32 = L.PW - 1, w16 = (m + 15) >> 4;
    uint32_t *q2 = sm + 4 * L.PW, *r2 = q2 + L.QW;
    for (int k = t; k < L.PW; k += nt) {
        uint32_t p0 = 0u, p1 = 0u, r0 = 0u, r1 = 0u, v = 0u;
        if (k < W32) {
            p0 = ldg(gq + 2 * k);
            r0 = ldg(gr + 2 * k);
            if (2 * k + 1 < w16) {
                p1 = ldg(gq + 2 * k + 1);
                r1 = ldg(gr + 2 * k + 1);
            }
            v = mask_below(m - 32 * k);
        }
        uint32_t lo, hi;
        planes_of(p0, p1, lo, hi);
        sm[k] = ~lo & ~hi & v;
        sm[L.PW + k] = lo & ~hi & v;
        sm[2 * L.PW + k] = ~lo & hi & v;
        sm[3 * L.PW + k] = lo & hi & v;
        q2[2 * k] = interleave_codes(p0);
        q2[2 * k + 1] = interleave_codes(p1);
        r2[2 * k] = interleave_codes(r0);
        r2[2 * k + 1] = interleave_codes(r1);
    }
}

// 16 two-bit codes from base j on.
SS_HD uint32_t code_window(const uint32_t *x, int j)
{
    return funnel_r(x[j >> 4], x[(j >> 4) + 1], (uint32_t)(2 * j) & 31u);
}

// Equal bases at the low end of two windows of codes (16: all).
SS_HD int code_run(uint32_t a, uint32_t b)
{
    const uint32_t x = a ^ b;
    const uint32_t y = (x | (x >> 1)) & 0x55555555u;
    return y ? (ffs32((int)y) - 1) >> 1 : 16;
}

// Farthest first obstacle over the starts of word i that `range` selects:
// rw and rw2 the codes of R[c .. c+15] and R[c+16 .. c+31], o[d] the plane
// offset of base R[c + d].
// TAIL: fewer than four columns are left from c.
template <bool TAIL>
SS_HD int team_word(const uint32_t *sm, const TeamLayout &L, int m, int c,
                    uint32_t rw, uint32_t rw2, const int (&o)[4], int i,
                    uint32_t range)
{
    const uint32_t *p = sm + i;
    const uint32_t S1 = p[o[0]] & range;
    uint32_t w1 = funnel_r(p[o[1]], p[o[1] + 1], 1);
    uint32_t w2 = funnel_r(p[o[2]], p[o[2] + 1], 2);
    uint32_t w3 = funnel_r(p[o[3]], p[o[3] + 1], 3);
    if (TAIL) {  // a row that reaches the row end stays
        w1 = c + 1 < m ? w1 : 0xffffffffu;
        w2 = c + 2 < m ? w2 : 0xffffffffu;
        w3 = c + 3 < m ? w3 : 0xffffffffu;
    }
    const uint32_t S2 = S1 & w1, S3 = S2 & w2;
    uint32_t S = S3 & w3;
    // no survivor: the column where the AND emptied
    int cand = c + (S1 ? 1 : 0) + (S2 ? 1 : 0) + (S3 ? 1 : 0);
    const uint32_t *q2 = sm + 4 * L.PW, *r2 = q2 + L.QW;
    while (S) {
        const int j = 32 * i + ffs32((int)S) - 1;
        S &= S - 1u;
        const int lim = m - imax(j, c);  // query or row end
        // two windows at once: most runs end in them
        const int a = code_run(code_window(q2, j), rw);
        const int b = code_run(code_window(q2, j + 16), rw2);
        int run = a < 16 ? a : 16 + b;
        if (run == 32) {
            while (run < lim) {
                const int k =
                    code_run(code_window(q2, j + run),
                             code_window(r2, c + run));
                run += k;
                if (k < 16)
                    break;
            }
        }
        cand = imax(cand, c + imin(run, lim));
    }
    return cand;
}

// The bits of word i >= lo/32 that are starts in lo..hi.
SS_HD uint32_t start_range(int i, int lo, int hi)
{
    return (0xffffffffu << imax(lo - 32 * i, 0)) &
           mask_below(hi + 1 - 32 * i);
}

#ifdef __CUDACC__
constexpr int kTeamWarps = 2;  // warps per CTA

// TEAM lanes per pair; a.slice_words shared words per pair.
template <int TEAM>
__global__ void __launch_bounds__(32 * kTeamWarps) k_cw_team(const CwArgs a)
{
    extern __shared__ uint32_t smem[];
    constexpr int PAIRS = 32 / TEAM;
    const int lane = threadIdx.x & 31, tl = lane % TEAM;
    uint32_t *sm = smem + (size_t)((threadIdx.x >> 5) * PAIRS + lane / TEAM) *
                              a.slice_words;
    const int begin = a.ws.ranges[2 * a.cls];
    const int end = a.ws.ranges[2 * a.cls + 1];
    bool alive = false, more = true;
    int64_t p = 0;
    int m = 1, E = 0, Ee = 0, c = 0, count = 0;
    TeamLayout L = TeamLayout::of(1);
    for (;;) {
        if (__any_sync(0xffffffffu, more && !alive)) {
            int idx = 0;
            if (more && !alive && tl == 0)
                idx = begin + (int)atomicAdd(&a.ws.counters[a.cls], 1u);
            idx = __shfl_sync(0xffffffffu, idx, 0, TEAM);
            if (more && !alive) {
                if (idx < end) {
                    p = a.ws.perm[idx];
                    m = a.ps.len(p);
                    E = a.ps.thr(p);
                    Ee = eff_threshold(m, E);
                    L = TeamLayout::of(m);
                    const int64_t off = a.ps.off(p);
                    team_stage(sm, L, a.ps.reads + off, a.ps.refs + off, m,
                               tl, TEAM);
                    count = 0;
                    alive = true;
                } else {
                    more = false;
                }
                c = 0;
            }
            __syncwarp();
        }
        if (!__any_sync(0xffffffffu, alive))
            break;
        const uint32_t *r2 = sm + 4 * L.PW + L.QW;
        // step until a team is done with its pair; tail: a team has fewer
        // than four columns left.  A team without a pair stays at column 0
        // with no starts.
        bool over = false;
        bool tail = __any_sync(0xffffffffu, alive && c + 4 > m);
        for (;;) {
            const uint32_t rw = code_window(r2, c);
            const uint32_t rw2 = code_window(r2, c + 16);
            int o[4];
#pragma unroll
            for (int d = 0; d < 4; ++d)
                o[d] = (int)((rw >> (2 * d)) & 3u) * L.PW;
            const int lo = max(c - Ee, 0), hi = min(c + Ee, m - 1);
            // the lane's word; past the window (or the query) no starts
            const int i = min((lo >> 5) + tl, L.PW - 1);
            const uint32_t range = alive ? start_range(i, lo, hi) : 0u;
            const int cand =
                tail ? team_word<true>(sm, L, m, c, rw, rw2, o, i, range)
                     : team_word<false>(sm, L, m, c, rw, rw2, o, i, range);
            int pstar;
            if constexpr (TEAM == 32) {
                pstar = __reduce_max_sync(0xffffffffu, cand);
            } else {
                pstar = cand;
#pragma unroll
                for (int s = TEAM / 2; s > 0; s >>= 1)
                    pstar = max(pstar, __shfl_xor_sync(0xffffffffu, pstar, s));
            }
            // an obstacle at pstar (perhaps on the last column), or the net
            // reached the destination
            if constexpr (TEAM == 32) {
                c = pstar + 1;
                count += pstar < m ? 1 : 0;
                over = c >= m || count > E;
                if (over)
                    break;
                tail = c + 4 > m;
            } else {
                c = alive ? pstar + 1 : 0;
                count += pstar < m ? 1 : 0;
                over = alive && (c >= m || count > E);
                if (!__any_sync(0xffffffffu, over || (alive && c + 4 > m)))
                    continue;
                if (__any_sync(0xffffffffu, over))
                    break;
                tail = true;
            }
        }
        if (over) {
            if (tl == 0) {
                a.ps.acc[p] = (uint8_t)(count <= E);
                a.ps.obs[p] = count;
            }
            alive = false;
            c = 0;
        }
        __syncwarp();  // the slice may be restaged
    }
}
#endif

}  // namespace ssk
