// ss_cwx.cuh -- K4 for thresholds from 817 (in served batches 512) to 10016:
// a CTA per pair, which looks the longest escape segments up in an index of
// the query instead of evaluating the maze rows; where that does not pay, it
// evaluates them.
//
// Method (Section 2.4): from checkpoint c the longest escape segment is the
// longest match of R[c..] with the query from any start j in c-E..c+E.  At
// E = 10^4 that is 20,001 rows, of which all but a few fail within eight
// columns; a start whose run is K or longer has Q[j..j+K) = R[c..c+K).  So
// the starts of each K-mer are kept in tables, and a column looks up its
// K-mer of R and extends only the starts found.
//
// The greedy is a chain (c -> c + run + 1), but what a column's longest run
// is does not depend on the chain: each of kIndexCols threads takes one of
// the next columns, while one more warp follows the chain through the
// results of the columns before, so a step costs a shared-memory load
// instead of the latency of its lookups.  (One warp per pair walking the
// chain lookup by lookup: 177 dependent instructions and 0.54 us a step; one
// CTA of 512 threads evaluating all rows with a barrier per step: 0.7 to 1.2
// us.)  What few columns need is done only where the chain stands on them:
//   * a thread compares a start over at most kIndexWindows windows; the
//     chain's warp extends a longer run, 512 bases per comparison;
//   * a column with several longer runs, or with more starts than a thread
//     is to go through, lies in a repeat: the CTA goes over to all rows;
//   * a column whose K-mer has no start in reach has a run shorter than K.
//     K-mers are numbered with the first base most significant, so the
//     starts of a shorter prefix are those of consecutive K-mers.
//
// The window c-E..c+E slides along the query, so the index is a ring of NB
// tables over blocks of BS consecutive starts: a counting sort of the
// block's starts by K-mer (4^K bucket ends, BS entries of 16 bits), built
// when the columns' windows reach the block, over the slot of a block they
// (and the chain's) have left: NB BS >= 2E + 2 kIndexCols + BS.  An entry
// holds the start and its next two bases, so 15 of 16 starts are dismissed
// without reading the query, as runs of K or K + 1.
// 1000 pairs of 10 to 100 kbp at E = 10 %: 11.2 -> 2.1 ms; the longest pair,
// 10^4 steps, is alone 1.8 ms of it (4 us per 224 columns, half lookups,
// half barrier and chain).
#pragma once
#include <cstdint>

#include "ss_bucket.cuh"
#include "ss_cw.cuh"
#include "ss_cws.cuh"
#include "ss_device.cuh"

namespace ssk {

constexpr int kIndexCols = 224;                // columns looked up at once
constexpr int kIndexThreads = kIndexCols + 32;  // and the chain's warp

// Index shape: K-mers, blocks of 2^LOGBS starts, NB tables; covers
// thresholds up to max_e().
template <int K_, int LOGBS_, int NB_, int COLS_ = kIndexCols>
struct IndexShape {
    static constexpr int K = K_, LOGBS = LOGBS_, NB = NB_, COLS = COLS_;
    static constexpr int BS = 1 << LOGBS;
    static constexpr int KMERS = 1 << (2 * K);
    static constexpr int SLOT = (KMERS + BS) / 2;  // 32-bit words per table
    static constexpr int WORDS = NB * SLOT;
    // the windows of 2 COLS columns, 2E + 2 COLS consecutive starts, touch
    // at most ceil((2E + 2 COLS - 1) / BS) + 1 blocks
    static constexpr int max_e() { return ((NB - 1) * BS - 2 * COLS) / 2; }
    static_assert(LOGBS <= 12, "an entry holds the start in 12 bits");
    static_assert(K >= 2 && K <= 14, "a K-mer and two bases in 32 bits");
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

// 16 bases, two bits each, the first in the two highest bits: from a packed
// word, and from the code bits of a window.
SS_HD uint32_t reverse_bits(uint32_t x)
{
#ifdef __CUDA_ARCH__
    return __brev(x);
#else
    uint32_t y = 0u;
    for (int i = 0; i < 32; ++i)
        y |= ((x >> i) & 1u) << (31 - i);
    return y;
#endif
}
SS_HD uint32_t bases_of_word(uint32_t w)
{
    return interleave_codes(reverse_bits(w));
}
SS_HD uint32_t bases_of_window(uint32_t lo, uint32_t hi)
{
    return interleave_codes((reverse_bits(lo) & 0xffff0000u) |
                            (reverse_bits(hi) >> 16));
}

// The K-mer that such bases start with, and (bits 12-15) the two bases
// after it, the first in the higher bits.
template <int K>
SS_HD uint32_t kmer_of(uint32_t bases)
{
    return bases >> (32 - 2 * K);
}
template <int K>
SS_HD uint32_t next_two(uint32_t bases)
{
    return ((bases << (2 * K)) >> 16) & 0xf000u;
}

// One more start of K-mer x in a table's counts (two 16-bit counts per
// word, none above BS): the count before.
SS_HD uint32_t table_add(uint32_t *tab, uint32_t x)
{
    const uint32_t sh = (x & 1u) * 16u;
#ifdef __CUDA_ARCH__
    const uint32_t old = atomicAdd(tab + (x >> 1), 1u << sh);
#else
    const uint32_t old = tab[x >> 1];
    tab[x >> 1] += 1u << sh;
#endif
    return (old >> sh) & 0xffffu;
}

// f(bases from the start on, start - first start of the block) for every
// start of block b that has K bases, by threads t, t + nt, ..., 16 starts
// each at a time.
template <class Sh, class F>
SS_HD void block_starts(const uint32_t *q, int w16, int m, int b, int t,
                        int nt, F f)
{
    const int j0 = b << Sh::LOGBS;
    const int j1 = imin(j0 + Sh::BS, m - Sh::K + 1);
    for (int j = j0 + 16 * t; j < j1; j += 16 * nt) {
        const int i = j >> 4;  // j is a multiple of 16
        const uint32_t a = bases_of_word(seq_word(q + i));
        const uint32_t z = i + 1 < w16 ? bases_of_word(seq_word(q + i + 1)) : 0u;
#pragma unroll
        for (int x = 0; x < 16; ++x)
            if (j + x < j1)
                f(funnel_l(z, a, 2 * x), j + x - j0);
    }
}

// Building the table of block b at tab (Sh::SLOT words: bucket ends, two
// per word, then the entries grouped by K-mer), thread t of nt; a barrier
// between the parts:
// 1. clear;
template <class Sh>
SS_HD void table_clear(uint32_t *tab, int t, int nt)
{
    for (int x = t; x < Sh::KMERS / 2; x += nt)
        tab[x] = 0u;
}
// 2. count the starts of each K-mer;
template <class Sh>
SS_HD void table_count(uint32_t *tab, const uint32_t *q, int w16, int m,
                       int b, int t, int nt)
{
    block_starts<Sh>(q, w16, m, b, t, nt, [&](uint32_t bases, int) {
        (void)table_add(tab, kmer_of<Sh::K>(bases));
    });
}
// 3. the thread's own words x0..x1 of the counts, their sum, and (after the
//    sums before it, run, are known) their exclusive prefixes;
template <class Sh>
SS_HD void table_span(int t, int nt, int &x0, int &x1)
{
    constexpr int HW = Sh::KMERS / 2;
    const int per = (HW + nt - 1) / nt;
    x0 = imin(t * per, HW);
    x1 = imin(x0 + per, HW);
}
template <class Sh>
SS_HD uint32_t table_sum(const uint32_t *tab, int t, int nt)
{
    int x0, x1;
    table_span<Sh>(t, nt, x0, x1);
    uint32_t sum = 0;
    for (int x = x0; x < x1; ++x)
        sum += (tab[x] & 0xffffu) + (tab[x] >> 16);
    return sum;
}
template <class Sh>
SS_HD void table_prefix(uint32_t *tab, uint32_t run, int t, int nt)
{
    int x0, x1;
    table_span<Sh>(t, nt, x0, x1);
    for (int x = x0; x < x1; ++x) {
        const uint32_t w = tab[x], mid = run + (w & 0xffffu);
        tab[x] = run | (mid << 16);
        run = mid + (w >> 16);
    }
}
// 4. scatter: each bucket's begin advances to its end.
template <class Sh>
SS_HD void table_scatter(uint32_t *tab, const uint32_t *q, int w16, int m,
                         int b, int t, int nt)
{
    uint16_t *entry = reinterpret_cast<uint16_t *>(tab + Sh::KMERS / 2);
    block_starts<Sh>(q, w16, m, b, t, nt, [&](uint32_t bases, int j) {
        entry[table_add(tab, kmer_of<Sh::K>(bases))] =
            (uint16_t)(j | next_two<Sh::K>(bases));
    });
}

// A column's result: the longest run found, 0 if no start shares its K-mer
// (the run is shorter than K); with kColumnOpen one start's run is not
// known to its end, and its row j - c + Ee is at bits 8 and up;
// kColumnRepeat: several starts' are not; kColumnMany: more starts share the
// K-mer, or agree with the column past it, than a thread looks at.
constexpr int kColumnOpen = 1 << 29, kColumnRepeat = 1 << 30;
constexpr int kColumnMany = kColumnRepeat + 1;
constexpr int kIndexWindows = 3;  // 51 to 96 bases of a start
// (random bases: two starts of a K-mer in a block at the most, five in reach,
// one in 16 of which agrees in the next two, where these are known)
constexpr int kIndexStarts = 24, kIndexExtends = 12;

// Longest match of R[c..] among the starts c-Ee..c+Ee in the tables.
template <class Sh>
SS_HD int column_longest(const uint32_t *tabs, const uint32_t *q,
                         const uint32_t *r, int w16, int m, int Ee, int c)
{
    constexpr int K = Sh::K;
    if (c + K > m)
        return 0;
    const int lo = imax(c - Ee, 0), hi = imin(c + Ee, m - 1);
    uint32_t rlo, rhi;
    int rn;
    base_window(r, w16, c, rlo, rhi, rn);
    const uint32_t bases = bases_of_window(rlo, rhi);
    const uint32_t k = kmer_of<K>(bases), want = next_two<K>(bases);
    int best = 0, open = 0;
    int extends = 0;
    int p0 = -1, p1 = -1;  // starts still to extend
    // (a start whose run is open: its row; false once there are two)
    auto extend = [&](int j) {
        const int run = index_run(q, r, w16, j, c, m - imax(j, c), rlo, rhi,
                                  rn, kIndexWindows);
        if (run < kRunOpen) {
            best = imax(best, run);
            return true;
        }
        const bool first = open == 0;
        open = kColumnOpen | (j - c + Ee) << 8;
        return first;
    };
    const int bh = hi >> Sh::LOGBS;
    for (int b = lo >> Sh::LOGBS; b <= bh; ++b) {
        const uint32_t *tab = tabs + (b % Sh::NB) * Sh::SLOT;
        const uint16_t *end = reinterpret_cast<const uint16_t *>(tab);
        const uint16_t *entry = end + Sh::KMERS;
        const int base = b << Sh::LOGBS;
        // where column or start have no two bases after their K-mer, the
        // entry's say nothing
        const uint32_t mask =
            imax(c, base + Sh::BS - 1) + K + 2 > m ? 0u : 0xf000u;
        const int e = end[k];
        int x = k ? end[k - 1] : 0;
        if (e - x > kIndexStarts)
            return kColumnMany;
        for (; x < e; ++x) {
            const uint32_t v = entry[x];
            const int j = base + (int)(v & 0xfffu);
            if ((uint32_t)(j - lo) > (uint32_t)(hi - lo))
                continue;
            const uint32_t d = (v ^ want) & mask;
            if (d != 0u) {
                best = imax(best, (d & 0xc000u) ? K : K + 1);
            } else if (p0 < 0) {
                p0 = j;
            } else if (p1 < 0) {
                p1 = j;
            } else if ((extends += mask ? 3 : 1) > kIndexExtends) {
                return kColumnMany;
            } else if (!extend(j)) {
                return kColumnRepeat;
            }
        }
    }
    if (p0 >= 0 && !extend(p0))
        return kColumnRepeat;
    if (p1 >= 0 && !extend(p1))
        return kColumnRepeat;
    return best | open;
}

// f(start) for every start in lo..hi whose K-mer is one of k0..k1, by lane
// t of nt (four to a table), until f returns false.
template <class Sh, class F>
SS_HD void bucket_starts(const uint32_t *tabs, uint32_t k0, uint32_t k1,
                         int lo, int hi, int t, int nt, F f)
{
    const int step = nt < 4 ? 1 : 4;
    for (int b = (lo >> Sh::LOGBS) + t / step; b <= hi >> Sh::LOGBS;
         b += nt / step) {
        const uint32_t *tab = tabs + (b % Sh::NB) * Sh::SLOT;
        const uint16_t *end = reinterpret_cast<const uint16_t *>(tab);
        const uint16_t *entry = end + Sh::KMERS;
        const int e = end[k1];
        for (int x = (k0 ? end[k0 - 1] : 0) + t % step; x < e; x += step) {
            const int j = (b << Sh::LOGBS) + (int)(entry[x] & 0xfffu);
            if (j >= lo && j <= hi && !f(j))
                return;
        }
    }
}

// Longest match of R[c..] of at least K bases, every start of its K-mer
// compared to the end (all lanes of a warp).
template <class Sh>
SS_HD int repeat_longest(const uint32_t *tabs, const uint32_t *q,
                         const uint32_t *r, int w16, int m, int Ee, int c,
                         int t, int nt)
{
    uint32_t rlo, rhi;
    int rn;
    base_window(r, w16, c, rlo, rhi, rn);
    const uint32_t k = kmer_of<Sh::K>(bases_of_window(rlo, rhi));
    int best = 0;
    bucket_starts<Sh>(tabs, k, k, imax(c - Ee, 0), imin(c + Ee, m - 1), t, nt,
                      [&](int j) {
                          best = imax(best, index_run(q, r, w16, j, c,
                                                      m - imax(j, c), rlo,
                                                      rhi, rn, 0));
                          return best < m - c;  // the row end: no farther
                      });
    return warp_max(best);
}

// Longest match of R[c..] where no start shares its K-mer, or fewer than K
// columns are left (all lanes of a warp): the longest prefix with a start in
// the tables, and the last starts, which have no K bases and are in no
// table.
template <class Sh>
SS_HD int short_longest(const uint32_t *tabs, const uint32_t *q,
                        const uint32_t *r, int w16, int m, int Ee, int c,
                        int t, int nt)
{
    constexpr int K = Sh::K;
    const int lo = imax(c - Ee, 0), hi = imin(c + Ee, m - 1);
    uint32_t rlo, rhi;
    int rn;
    base_window(r, w16, c, rlo, rhi, rn);
    const uint32_t bases = bases_of_window(rlo, rhi);
    int best = 0;
    for (int j = imax(m - K + 1, lo) + t; j <= hi; j += nt)
        best = imax(best, index_run(q, r, w16, j, c, m - imax(j, c), rlo,
                                    rhi, rn, 0));
    best = warp_max(best);
    for (int l = imin(K - 1, m - c); l > best; --l) {
        const uint32_t k0 = (bases >> (32 - 2 * l)) << (2 * (K - l));
        int any = 0;
        bucket_starts<Sh>(tabs, k0, k0 + (1u << (2 * (K - l))) - 1u, lo, hi,
                          t, nt, [&](int) {
                              any = 1;
                              return false;
                          });
        if (warp_max(any))
            return l;
    }
    return best;
}

// The chain's state; done: 1 at its end, kChainMany on a column with too many
// starts (if it stops there).
struct IndexChain {
    int c, count, done;
};
constexpr int kChainMany = 2;

// Follow the chain from s.c through the columns c0..c0+cols-1, whose
// results are in col[] (all lanes of a warp, with the same state): one
// obstacle after each run (Section 2.4 steps 3 and 4).  many: stop at a column
// with more starts than kIndexRepeat (else the warp compares all of them).
template <class Sh>
SS_HD void chain_follow(IndexChain &s, const int *col, int c0, int cols,
                        const uint32_t *tabs, const uint32_t *q,
                        const uint32_t *r, int w16, int m, int E, int Ee,
                        int t, int nt, bool many = false)
{
    while (!s.done && s.c - c0 < cols) {
        const int v = col[s.c - c0];
        int run = v & 0xff;
        if (v & kColumnOpen) {
            const int j = ((v & (kColumnOpen - 1)) >> 8) - Ee + s.c;
            run = imax(run, warp_run(q, r, w16, j, s.c, m - imax(j, s.c)));
        } else if (v >= kColumnRepeat && many) {
            s.done = kChainMany;
            return;
        } else if (v >= kColumnRepeat) {
            run = repeat_longest<Sh>(tabs, q, r, w16, m, Ee, s.c, t, nt);
        } else if (v == 0) {
            run = short_longest<Sh>(tabs, q, r, w16, m, Ee, s.c, t, nt);
        }
        if (s.c + run >= m) {
            s.done = 1;  // the net reached the destination
        } else {
            ++s.count;
            s.c += run + 1;
            // past E, or the obstacle stood on the last column
            s.done = s.count > E || s.c >= m;
        }
    }
}

// ---- all rows ----------------------------------------------------------------
//
// What the index does not answer cheaply -- columns whose K-mer has many
// starts, as in a repeat, and pairs whose steps are so long that most columns
// looked up are never stood on -- the CTA routes by all rows (ss_cws.cuh), 32
// to a thread, whatever the bases; then the index goes on.  Ms, the index
// alone / with all rows / a CTA over all rows from the start, the whole pair
// staged: 20 pairs of 10 to 100 kbp of a dinucleotide repeat with 5 % errors,
// E = 10 %, 830 / 10.4 / 9.2; of a 171-base repeat 16.6 / 7.3 / 5.5; 1000 of
// it of 10 to 30 kbp 3.7 / 2.1 / 2.1; 152 pairs of 100 kbp, E = 1 %, 0.8 %
// errors 1.5 / 0.64 / 0.65, E = 10 %, 8 % errors 2.0 / 2.1 / 6.0.

// The rings of a CTA of THREADS threads that takes one pair.
template <int QB_, int RB_, int THREADS_>
struct RowsShape {
    static constexpr int QB = QB_, RB = RB_, BP = 1024, LANES = THREADS_;
    static constexpr int QW = QB / 32, RW = RB / 32;
    static constexpr int AHEAD = 32 * 32 + 95;  // a warp follows a row
    static constexpr int WORDS = 2 * (QW + 1 + RW + 1);
    static constexpr int max_e() { return (QB - BP - AHEAD - 1) / 2; }
    static_assert(RB >= BP + AHEAD + 1, "a step in the reference's ring");
};

// The classes' shapes: one to five starts per K-mer and window.
using IndexShape0 = IndexShape<5, 11, 3>;  // E' <= 1664:   18 KB
using IndexShape1 = IndexShape<6, 12, 4>;  // E' <= 5920:   64 KB
using IndexShape2 = IndexShape<6, 12, 6>;  // E' <= 10016:  96 KB

static_assert(IndexShape0::max_e() >= index_max_e(0) &&
                  IndexShape1::max_e() >= index_max_e(1) &&
                  IndexShape2::max_e() >= index_max_e(2),
              "a class's thresholds fit its tables");

// STEPS: as many steps by all rows take as long as a turn of kIndexCols columns
// (a pair alone: 0.34 us each at E' = 1000, 0.6 at 5000, 1.2 at 10^4, against
// 2.5, 3.0 and 4.0 a turn).
template <int C>
struct IndexClass;
template <>
struct IndexClass<0> {
    using Shape = IndexShape0;
    using Rows = RowsShape<16384, 8192, kIndexThreads>;
    static constexpr int STEPS = 4;
};
template <>
struct IndexClass<1> {
    using Shape = IndexShape1;
    using Rows = RowsShape<16384, 8192, kIndexThreads>;
    static constexpr int STEPS = 3;
};
template <>
struct IndexClass<2> {
    using Shape = IndexShape2;
    using Rows = RowsShape<32768, 8192, kIndexThreads>;
    static constexpr int STEPS = 2;
};

// Shared words of a CTA of index class C: the tables, or in their place the
// rings of all rows.  (Rings beside the tables would save building them again,
// but left room for fewer CTAs on an SM: 1000 pairs of 10 to 100 kbp at 10 %
// 2.15 -> 2.4 ms.)
template <int C>
constexpr int index_smem_words()
{
    static_assert(IndexClass<C>::Rows::max_e() >= index_max_e(C),
                  "a class's thresholds fit its rings");
    static_assert(IndexClass<C>::Rows::WORDS <= IndexClass<C>::Shape::WORDS,
                  "the rings in the tables' place");
    return IndexClass<C>::Shape::WORDS;
}

// Pairs whose obstacles, if they use up E, are on average more than this many
// columns apart begin by all rows.
constexpr int kIndexSparse = 32;

#ifdef __CUDACC__
constexpr int kRowsWarps = kIndexThreads / 32;
struct RowsShared {
    int best[2][kRowsWarps];
    IndexChain chain;
};

// What the threads of a CTA share besides the tables.
struct IndexShared {
    int col[2][kIndexCols];  // the columns' results
    uint32_t part[kIndexCols / 32];
    IndexChain chain;
    RowsShared rows;
};

// Barrier of the kIndexCols threads that look columns up.
__device__ __forceinline__ void cols_sync()
{
    asm volatile("bar.sync 1, %0;" : : "n"(kIndexCols) : "memory");
}

// Build the table of block b (threads 0..kIndexCols-1).
template <class Sh>
__device__ __forceinline__ void build_table(uint32_t *tab, IndexShared &s,
                                            const uint32_t *q, int w16, int m,
                                            int b)
{
    const int t = threadIdx.x, nt = kIndexCols;
    table_clear<Sh>(tab, t, nt);
    cols_sync();
    table_count<Sh>(tab, q, w16, m, b, t, nt);
    cols_sync();
    const uint32_t sum = table_sum<Sh>(tab, t, nt);
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
        if ((t & 31) >= o)
            incl += v;
    }
    if ((t & 31) == 31)
        s.part[t >> 5] = incl;
    cols_sync();
    uint32_t run = incl - sum;
    for (int w = 0; w < t >> 5; ++w)
        run += s.part[w];
    table_prefix<Sh>(tab, run, t, nt);
    cols_sync();
    table_scatter<Sh>(tab, q, w16, m, b, t, nt);
    cols_sync();
}

// Barrier of the CTA's first n threads.
__device__ __forceinline__ void rows_sync(int n)
{
    asm volatile("bar.sync 2, %0;" : : "r"(n) : "memory");
}

// Maximum over the first n threads of v, the same in the lanes of a warp
// (best: a buffer their next call does not use).
__device__ __forceinline__ int rows_best(int (&best)[kRowsWarps], int n, int v)
{
    const int lane = threadIdx.x & 31;
    if (lane == 0)
        best[threadIdx.x >> 5] = v;
    rows_sync(n);
    return __reduce_max_sync(0xffffffffu, lane < n >> 5 ? best[lane] : 0);
}

// Follow the chain of a pair from s.c by all rows, until its end or until
// the index would be faster: for `calm` stretches of kRowsStretch columns in
// a row no lane had many survivors, and the last one's steps were of fewer
// than `dense` columns each; x: Sh::WORDS words.  As many of the CTA's warps
// take part as the window has words for.  (With half as many and two words a
// lane 152 pairs of 100 kbp at E' = 1500 took 950 us instead of 790.)
constexpr int kRowsStretch = 2048;
template <class Sh>
__device__ __noinline__ void rows_route(uint32_t *x, RowsShared &sh,
                                        IndexChain &chain, const uint32_t *q,
                                        const uint32_t *r, int m, int E,
                                        int Ee, int calm, int dense)
{
    const int t = threadIdx.x;
    const int nt = min((2 * Ee + 1 + 1023) >> 10, Sh::LANES / 32) * 32;
    if (t < nt) {
        uint2 *q2 = reinterpret_cast<uint2 *>(x), *r2 = q2 + Sh::QW + 1;
        RingStep s;
        s.q2 = q2;
        s.r2 = r2;
        s.q = q;
        s.r = r;
        s.m = m;
        s.w16 = (m + 15) >> 4;
        s.c = chain.c;
        int count = chain.count, qn = 0, rn = 0, buf = 0, quiet = 0;
        bool over = false;
        while (!over) {
            // fill the rings as far as they go
            qn = max(qn, max(s.c - Ee, 0) & ~(Sh::BP - 1));
            rn = max(rn, s.c & ~(Sh::BP - 1));
            const int q0 = qn, r0 = rn;
            while (ring_room(qn, m, s.c - Ee, Sh::QB, Sh::BP))
                qn += Sh::BP;
            while (ring_room(rn, m, s.c, Sh::RB, Sh::BP))
                rn += Sh::BP;
            ring_fill<Sh::QW>(q2, q, s.w16, q0, qn, t, nt);
            ring_fill<Sh::RW>(r2, r, s.w16, r0, rn, t, nt);
            const int until = min(min(ring_until(qn, m, Ee + Sh::AHEAD),
                                      ring_until(rn, m, Sh::AHEAD)),
                                  s.c + kRowsStretch);
            rows_sync(nt);
            const int c0 = s.c, count0 = count;
            bool many = false;
            do {
                ring_window<Sh::RW>(r2, s.c, s.rlo, s.rhi);
                s.lo = max(s.c - Ee, 0);
                s.hi = min(s.c + Ee, m - 1);
                int best = rows_best(sh.best[buf], nt,
                                     rows_step<Sh>(s, t, 32 * nt, many));
                buf ^= 1;
                if (best < 4) {
                    int pre = 0;
                    for (int i = (s.lo >> 5) + t; i <= s.hi >> 5; i += nt)
                        pre = max(pre, prefix_word<Sh>(s, m - s.c, i));
                    best = rows_best(sh.best[buf], nt, warp_max(pre));
                    buf ^= 1;
                }
                s.c += best + 1;
                count += s.c <= m ? 1 : 0;
                over = s.c >= m || count > E;
            } while (!over && s.c < until);
            // (the barrier also lets the rings be written again)
            const int any = rows_best(sh.best[buf], nt,
                                      __any_sync(0xffffffffu, many));
            buf ^= 1;
            quiet = any ? 0 : quiet + 1;
            if (quiet >= calm && s.c - c0 < dense * (count - count0))
                over = true;
        }
        if (t == 0)
            sh.chain = IndexChain{s.c, count, s.c >= m || count > E};
    }
    __syncthreads();
    chain = sh.chain;
    __syncthreads();  // sh.chain is written again
}

// Route one pair with the CTA's kIndexThreads threads; smem:
// index_smem_words<C>() words.  Returns min(count, E+1) to every thread.
// Ee = eff_threshold(m, E) <= max_e().
template <int C>
__device__ __noinline__ int index_route(uint32_t *smem, IndexShared &s,
                                        const uint32_t *q, const uint32_t *r,
                                        int m, int E)
{
    using Sh = typename IndexClass<C>::Shape;
    using Rows = typename IndexClass<C>::Rows;
    uint32_t *tabs = smem, *rings = smem;  // one or the other
    const int t = threadIdx.x;
    const int Ee = eff_threshold(m, E), w16 = (m + 15) >> 4;
    constexpr int STEPS = IndexClass<C>::STEPS;
    constexpr int DENSE = kIndexCols / (2 * STEPS);
    int built = 0, buf = 0;
    int calm = 1;  // quiet stretches by all rows before the index goes on
    int steps = 8 * STEPS;       // of the last turns, their mean four times
    int before = 0;              // obstacles before a turn
    // columns at..: being looked up into col[buf]; those at c0..: in
    // col[buf ^ 1], for the chain (none in the first turn)
    int at = 0, c0 = -kIndexCols;
    IndexChain chain{0, 0, 0};
    bool rows = (int64_t)Ee * kIndexSparse < m;
    for (;;) {
        if (rows) {
            rows_route<Rows>(rings, s.rows, chain, q, r, m, E, Ee, calm,
                             DENSE);
            if (chain.done)
                return chain.count;
            // (the columns looked up ahead are dropped, the tables built again)
            rows = false;
            built = 0;
            steps = 8 * STEPS;
            before = chain.count;
            at = chain.c;
            c0 = at - kIndexCols;
        }
        if (t < kIndexCols) {
            const int last = min(at + kIndexCols - 1 + Ee, m - 1);
            // (blocks that a long run passed over are not built)
            built = max(built, max(at - Ee, 0) >> Sh::LOGBS);
            for (; at < m && built <= last >> Sh::LOGBS; ++built)
                build_table<Sh>(tabs + (built % Sh::NB) * Sh::SLOT, s, q, w16,
                                m, built);
            s.col[buf][t] =
                column_longest<Sh>(tabs, q, r, w16, m, Ee, at + t);
        } else {
            chain_follow<Sh>(chain, s.col[buf ^ 1], c0, kIndexCols, tabs, q,
                             r, w16, m, E, Ee, t - kIndexCols, 32, true);
            if (t == kIndexCols)
                s.chain = chain;
        }
        __syncthreads();
        chain = s.chain;
        if (chain.done == 1)
            return chain.count;
        if (chain.done == kChainMany) {
            // a repeat: by all rows until it is over, longer each time
            chain.done = 0;
            calm = min(2 * calm, 64);
            rows = true;
            continue;
        }
        // steps so long that most columns are looked up in vain
        if (c0 >= 0)
            steps += chain.count - before - (steps >> 2);
        before = chain.count;
        rows = steps < 4 * STEPS;
        c0 = at;
        // the chain may have left these columns behind already
        at = max(at + kIndexCols, chain.c);
        buf ^= 1;
        __syncthreads();  // s.chain is written again
    }
}

// Route a pair of index class ic, or (above them) of any threshold: by all
// rows, the whole query in the ring.
using WholeRows = RowsShape<131072, 8192, kIndexThreads>;
static_assert(WholeRows::QB >= kMaxLen &&
                  WholeRows::WORDS <= index_smem_words<2>(),
              "the longest query in the ring, in the tables' place");
__device__ __forceinline__ int index_route_any(int ic, uint32_t *smem,
                                               IndexShared &s,
                                               const uint32_t *q,
                                               const uint32_t *r, int m,
                                               int E)
{
    switch (ic) {
    case 0: return index_route<0>(smem, s, q, r, m, E);
    case 1: return index_route<1>(smem, s, q, r, m, E);
    case 2: return index_route<2>(smem, s, q, r, m, E);
    default: break;
    }
    IndexChain chain{0, 0, 0};
    rows_route<WholeRows>(smem, s.rows, chain, q, r, m, E,
                          eff_threshold(m, E), 1, 0);
    return chain.count;
}

// A pair at a time from the class's queue.
template <int C>
__global__ void __launch_bounds__(kIndexThreads, C == 0 ? 4 : 3)
    k_cw_index(const CwArgs a)
{
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ IndexShared s;
    __shared__ int s_idx;
    const int t = threadIdx.x;
    const int begin = a.ws.ranges[2 * a.cls];
    const int end = a.ws.ranges[2 * a.cls + 1];
    if (a.queued && long_queued(a.cls))
        return;  // routed by the serving queue's worker
    // the first without waiting for the counter (in the order of their
    // claims, few pairs stood two on every other SM)
    for (int idx = begin + (int)blockIdx.x; idx < end;) {
        const int64_t p = a.ws.perm[idx];
        const int m = a.ps.len(p), E = a.ps.thr(p);
        const int64_t off = a.ps.off(p);
        const int count = index_route<C>(smem, s, a.ps.reads + off,
                                         a.ps.refs + off, m, E);
        if (t == 0) {
            a.ps.acc[p] = (uint8_t)(count <= E);
            a.ps.obs[p] = count;
            s_idx = begin + (int)gridDim.x +
                    (int)atomicAdd(&a.ws.counters[a.cls], 1u);
        }
        __syncthreads();
        idx = s_idx;
        __syncthreads();  // the tables and s_idx are reused
    }
}
#endif

}  // namespace ssk
