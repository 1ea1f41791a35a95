// ss_pm.cuh -- pair-major packed batches (SS_FMT_PACKED2, uniform m) walked
// bit-sliced, 32 pairs per thread, without a sliced copy in memory: a warp
// stages up to 32 groups of 32 pairs in shared memory, and each lane turns
// its own group into bit-sliced words in place, and walks it from there
// (ss_sliced.cuh).
//
// Why: a pair costs a thread of its own some ops per cell or column, the
// walk of 32 pairs per word a 32nd of that, and turning 32 words of 16 bases
// costs about 210 ops, 6.5 per word and pair: 91 a pair of 100 bp.
// Staging: 4-byte asynchronous copies, 32 consecutive words of a group at a
// time, each to its place, so that the 16 bases' words of a group's 32 pairs
// end up side by side; the turn and the walk then read and write one lane's
// region, whose stride is odd, without bank conflicts, and no lane exchanges
// anything with another.  (With lane i copying pair i's words a copy touched
// about w16 + 1 lines: exact distances of 3M pairs of 100 bp, E = 0 / 5 93 /
// 112 -> 83 / 102 us, 1.2M of 250 bp 151 / 210 -> 118 / 178, sub-mazes of 3M
// of 100 bp, E = 5 137 -> 127.)
// One warp per CTA and up to 56 KB of shared memory, so that four CTAs stand
// on an SM, one per scheduler: a pair's 2 bits per base set how many can be
// in flight, so a walk lives from the independence of its rows, and the
// staging of one CTA overlaps the walks of the others.  Bound by the issue
// of one warp per scheduler: 0.31 to 0.36 instructions a cycle (E = 0 and 5),
// where the logic pipe takes one every two, and a sixth of the time waits for
// the staged words.
// What else was measured, exact distances of 3M pairs of 100 bp at E = 0 /
// 31 (this form, before the copies went by lines: 92 / 233 us): words copied as they lie in memory and turned
// in their places, every later address a multiple of w16: 140 / 281; two
// warps per CTA, one side each, then one walking (the walking warps of all
// CTAs on two schedulers): 93 / 354; words turned in registers, 16 bases at
// a time, as the walk reaches them (2000 instructions without a loop): 124 /
// 367.
#pragma once
#include <cstdint>

#include "ss_device.cuh"
#include "ss_sliced.cuh"

namespace ssk {

// 32 x 32 bits transposed in place: bit i of a[r] becomes what bit r of a[i]
// was (a[i] the word of pair i; a[r] then bit r of all pairs).
SS_HD void transpose32(uint32_t (&a)[32])
{
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const uint32_t x = a[k], y = a[k + 16];
        a[k] = prmt(x, y, 0x5410u);
        a[k + 16] = prmt(x, y, 0x7632u);
    }
#pragma unroll
    for (int h = 0; h < 32; h += 16)
#pragma unroll
        for (int k = h; k < h + 8; ++k) {
            const uint32_t x = a[k], y = a[k + 8];
            a[k] = prmt(x, y, 0x6240u);
            a[k + 8] = prmt(x, y, 0x7351u);
        }
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        const int d = 4 >> l;
        const uint32_t M = d == 4 ? 0x0f0f0f0fu
                                  : d == 2 ? 0x33333333u : 0x55555555u;
#pragma unroll
        for (int k = 0; k < 32; ++k) {
            if (k & d)
                continue;
            const uint32_t x = a[k], y = a[k + d];
            a[k] = lop3<0xE4>(x, y << d, M);      // (x & M) | (y << d & ~M)
            a[k + d] = lop3<0xE4>(x >> d, y, M);  // (x >> d & M) | (y & ~M)
        }
    }
}

// Words of one group's region per side: w16 chunks of 32 words (one word per
// pair, later one per code bit and base), and one to make the stride odd.
SS_HD int pm_stride(int w16) { return 32 * w16 + 1; }

// Where a region holds word c of its pair i until the turn: the words of
// consecutive pairs are copied side by side, and would fall w16 to a bank
// (32c + i); fours of pairs change places by c, which leaves about two.
SS_HD int pm_place(int c, int i) { return 32 * c + (i ^ (4 * (c & 7))); }

// Turn a region's w16 chunks into bit-sliced words: word 32c + 16b + t is
// code bit b of base 16c + t, one pair per bit.
SS_HD void pm_turn(uint32_t *x, int w16)
{
    for (int c = 0; c < w16; ++c) {
        uint32_t a[32];
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
            const uint32_t *p = x + pm_place(c, i);
            a[i] = p[0];
            a[i + 1] = p[1];
            a[i + 2] = p[2];
            a[i + 3] = p[3];
        }
        transpose32(a);
#pragma unroll
        for (int i = 0; i < 32; ++i)
            x[32 * c + i] = a[i];
    }
}

// A turned pair of regions as the walks read it (four bases per block).
struct PmSrc {
    const uint32_t *q, *r;
    SS_HD static void load(const uint32_t *x, int blk, uint32_t (&lo)[4],
                           uint32_t (&hi)[4])
    {
        const uint32_t *p = x + (blk >> 2) * 32 + (blk & 3) * 4;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            lo[k] = p[k];
            hi[k] = p[16 + k];
        }
    }
    SS_HD void query(int blk, int nb, uint32_t (&lo)[4],
                     uint32_t (&hi)[4]) const
    {
        if (blk < 0 || blk >= nb) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                lo[k] = hi[k] = 0u;
            return;
        }
        load(q, blk, lo, hi);
    }
    SS_HD void ref(int blk, uint32_t (&lo)[4], uint32_t (&hi)[4]) const
    {
        load(r, blk, lo, hi);
    }
    SS_HD void prefetch(int, int, int, int) const {}
};

// ---- exact distances -------------------------------------------------------
//
// min(ED, E+1) of 32 pairs at once: the table of the Levenshtein distance
// by its differences (Myers 1999), one bit per pair.  For cell (i, j) with
// eq = [Q_i == R_j], the vertical difference at its left (+1: Pv, -1: Mv)
// and the horizontal one above it (Ph, Mh):
//     D0 = eq | Mv | Mh                       (diagonal difference 0)
//     Ph' = Mv | ~(D0 | Pv),  Mh' = D0 & Pv   (horizontal, below)
//     Pv' = Mh | ~(D0 | Ph),  Mv' = D0 & Ph   (vertical, at its right)
// -- seven three-input ops per cell and 32 pairs.  A path of at most E edits
// that returns to the main diagonal strays at most E/2 from it, so the band
// is H = E/2 diagonals either side (rounded down): E+1 cells per row instead
// of 2E+1; outside it neighbours count as one more (they never help).  The
// distance is the number of diagonal differences 1 on the main diagonal.
template <int E>
struct EdShape {
    static constexpr int H = E / 2;
    static constexpr int ND = 2 * H + 1;
    static constexpr int NBH = (H + 3) / 4;       // window blocks per side
    static constexpr int WW = 4 * (2 * NBH + 1);  // window words per plane
};

// Row x (read base x, words qlo, qhi) of the band; wl, wh: the window of the
// reference, word w = base j0 - 4 NBH + w of the block j0..j0+3, x = j0 + U.
// EDGE: reference bases before the first match nothing.
template <int E, bool EDGE, int U>
SS_HD void ed_row(uint32_t (&Ph)[EdShape<E>::ND], uint32_t (&Mh)[EdShape<E>::ND],
                  SlicedCount<E> &cnt, const uint32_t (&wl)[EdShape<E>::WW],
                  const uint32_t (&wh)[EdShape<E>::WW], uint32_t qlo,
                  uint32_t qhi, int x)
{
    using Sh = EdShape<E>;
    uint32_t Pv = 0xffffffffu, Mv = 0u;
#pragma unroll
    for (int d = 0; d < Sh::ND; ++d) {
        const int w = 4 * Sh::NBH - Sh::H + U + d;
        uint32_t eq = lop3<0x90>(~(wl[w] ^ qlo), wh[w], qhi);
        if (EDGE)
            eq = x + d - Sh::H >= 0 ? eq : 0u;
        const uint32_t ph = d + 1 < Sh::ND ? Ph[d + 1] : 0xffffffffu;
        const uint32_t mh = d + 1 < Sh::ND ? Mh[d + 1] : 0u;
        const uint32_t D0 = lop3<0xFE>(eq, Mv, mh);
        Ph[d] = lop3<0xF1>(Mv, D0, Pv);  // a | ~(b | c)
        Mh[d] = D0 & Pv;
        Pv = lop3<0xF1>(mh, D0, ph);
        Mv = D0 & ph;
        if (d == Sh::H)
            cnt.step(D0);
    }
}

// min(ED, E+1) of a group's pairs of length m; src.query the reads, src.ref
// the references; pad: pairs that do not exist.
template <int E, class Src>
SS_HD void ed_walk(const Src &src, int m, uint32_t pad, SlicedCount<E> &cnt)
{
    using Sh = EdShape<E>;
    const int nb = (m + 3) >> 2;
    uint32_t wl[Sh::WW], wh[Sh::WW];
    // the window is over the references: Src's bounds-checked loads are its
    // query's
    const Src ref{src.r, src.q};
#pragma unroll
    for (int b = 0; b < 2 * Sh::NBH + 1; ++b) {
        uint32_t lo[4], hi[4];
        ref.query(b - Sh::NBH, nb, lo, hi);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            wl[4 * b + k] = lo[k];
            wh[4 * b + k] = hi[k];
        }
    }
    uint32_t Ph[Sh::ND], Mh[Sh::ND];
#pragma unroll
    for (int d = 0; d < Sh::ND; ++d) {
        Ph[d] = d > Sh::H ? 0xffffffffu : 0u;  // D[0][j] = j
        Mh[d] = 0u;
    }
    cnt.init(pad);
    for (int k = 0; k < nb; ++k) {
        uint32_t ql[4], qh[4];
        ref.ref(k, ql, qh);
        const int x = 4 * k, live = m - x;
        auto rows = [&](auto edge) {
            constexpr bool EDGE = decltype(edge)::value;
            ed_row<E, EDGE, 0>(Ph, Mh, cnt, wl, wh, ql[0], qh[0], x);
            if (live > 3) {
                // (no branch between rows: a row's chain along the band
                // runs beside the next row's)
                ed_row<E, EDGE, 1>(Ph, Mh, cnt, wl, wh, ql[1], qh[1], x + 1);
                ed_row<E, EDGE, 2>(Ph, Mh, cnt, wl, wh, ql[2], qh[2], x + 2);
                ed_row<E, EDGE, 3>(Ph, Mh, cnt, wl, wh, ql[3], qh[3], x + 3);
                return;
            }
            if (live > 1)
                ed_row<E, EDGE, 1>(Ph, Mh, cnt, wl, wh, ql[1], qh[1], x + 1);
            if (live > 2)
                ed_row<E, EDGE, 2>(Ph, Mh, cnt, wl, wh, ql[2], qh[2], x + 2);
        };
        if (x < Sh::H)
            rows(std::true_type{});
        else
            rows(std::false_type{});
        if (cnt.done() == 0xffffffffu)
            return;  // every pair past E
        uint32_t lo[4], hi[4];
        ref.query(k + Sh::NBH + 1, nb, lo, hi);
#pragma unroll
        for (int w = 0; w + 4 < Sh::WW; ++w) {
            wl[w] = wl[w + 4];
            wh[w] = wh[w + 4];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            wl[Sh::WW - 4 + i] = lo[i];
            wh[Sh::WW - 4 + i] = hi[i];
        }
    }
}

#ifdef __CUDACC__
// Shared memory per CTA, so that four stand on an SM (228 KB, 1 KB of each
// reserved) beside `fixed` bytes of the kernel's own.
constexpr int kPmSmem = 56 * 1024;
constexpr size_t pm_budget(size_t fixed)
{
    return fixed < 1024 ? (size_t)kPmSmem - 512 : (size_t)kPmSmem - fixed;
}

struct PmArgs {
    const uint32_t *q, *r;  // pair p at word p * w16
    int64_t n;
    int32_t m, w16;
    int32_t G;              // groups per CTA (1..32)
    uint32_t one;           // 1 (see sliced_column)
};

constexpr int kPmThreads = 32;

// Stage G groups of both sides, the reads' regions at x, the references'
// after them (q, r: the words of the first group's pairs, pairs of them
// exist): a group's words as they follow one another in memory, 32 per copy;
// words of pairs that do not exist are zero.
__device__ __forceinline__ void pm_stage(uint32_t *x, const uint32_t *q,
                                         const uint32_t *r, int64_t pairs,
                                         int G, int w16)
{
    const int lane = threadIdx.x, stride = pm_stride(w16);
    const int full = (int)min((int64_t)G, pairs >> 5);
    const int du = 32 / w16, dc = 32 % w16;
    int u = lane / w16, c = lane % w16;  // word 32k + lane: pair, word of it
    for (int k = 0; k < w16; ++k) {
        uint32_t *to = x + pm_place(c, u);
        uint32_t at = smem_addr(to);
        int from = 32 * k + lane;
#pragma unroll 4
        for (int g = 0; g < full; ++g) {
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(at),
                         "l"(q + from)
                         : "memory");
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                             at + 4 * G * stride),
                         "l"(r + from)
                         : "memory");
            at += 4 * stride;
            from += 32 * w16;
        }
        // the batch's last pairs, and groups past it
        for (int g = full; g < G; ++g) {
            const bool exists = 32 * g + u < pairs;
            const int at_word = (32 * g + u) * w16 + c;
            to[g * stride] = exists ? q[at_word] : 0u;
            to[(G + g) * stride] = exists ? r[at_word] : 0u;
        }
        u += du;
        c += dc;
        if (c >= w16) {
            c -= w16;
            ++u;
        }
    }
}

// Stage the CTA's groups and turn them, a group per lane; false for a lane
// without a group.
__device__ __forceinline__ bool pm_prepare(uint32_t *x, const PmArgs &a,
                                           PmSrc &src, int64_t &p0, int &np)
{
    const int lane = threadIdx.x, stride = pm_stride(a.w16);
    const int64_t first = (int64_t)blockIdx.x * a.G * 32;
    pm_stage(x, a.q + first * a.w16, a.r + first * a.w16, a.n - first, a.G,
             a.w16);
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::
                     : "memory");
    __syncwarp();
    p0 = first + 32 * lane;
    if (lane >= a.G || p0 >= a.n)
        return false;
    np = (int)min((int64_t)32, a.n - p0);
    uint32_t *q = x + lane * stride, *r = q + a.G * stride;
    pm_turn(q, a.w16);
    pm_turn(r, a.w16);
    src = PmSrc{q, r};
    return true;
}

// Fill a and the launch shape for n pairs of m bases: as many groups per
// CTA as the shared memory holds, fewer where the batch leaves SMs idle.
// False where a single group does not fit.
inline bool pm_config(const uint32_t *q, const uint32_t *r, int64_t n,
                      int32_t m, int sm_count, size_t fixed, PmArgs &a,
                      unsigned &grid, size_t &smem)
{
    a.q = q;
    a.r = r;
    a.n = n;
    a.m = m;
    a.w16 = (m + 15) / 16;
    a.one = 1u;
    const size_t per = (size_t)2 * (size_t)pm_stride(a.w16) * 4;
    if (m <= 0 || n <= 0 || per > pm_budget(fixed))
        return false;
    const int64_t groups = (n + 31) / 32;
    const int64_t spread = (groups + 4 * sm_count - 1) / (4 * sm_count);
    int64_t G = (int64_t)(pm_budget(fixed) / per);
    G = G < 32 ? G : 32;
    G = G < spread ? G : spread;
    a.G = (int32_t)(G > 0 ? G : 1);
    const int64_t blocks = (groups + a.G - 1) / a.G;
    if (blocks > 0x7fffffff)
        return false;
    grid = (unsigned)blocks;
    smem = per * a.G;
    return true;
}
#endif

}  // namespace ssk
