// ss_bucket.cuh -- K2: length/threshold buckets of a mixed batch, and the
// per-pair accessors shared by the bucketed kernels.
//
// Every pair is assigned to one class -- which kernel routes it -- from its
// length m and effective threshold E' = min(E, m-1) (rows with |s| >= m hold
// no Q base at all, so they are all obstacles and never bound the longest
// run; the count limit still uses E):
//   * RW classes: E' <= 31, thread per pair, E' <= EMAX in {1, 3, 7, 15, 31}
//   * ring classes: E' <= 816, a team of 2 or 4 lanes or (few pairs,
//     repeats) a warp per pair (ss_cws.cuh), by E'
//   * index classes: E' <= 10016, CTA per pair (ss_cwx.cuh), by E'
//   * CTA classes: larger E', CTA per pair (ss_cw.cuh), by m bound
// Within a class pairs are ordered by length, longest first (quarter-octave
// bins), so that persistent workers take the biggest pairs first and a warp
// of the RW kernel sees similar lengths.
#pragma once
#include <cstdint>

#include "ss_rw_config.h"

namespace ssk {

constexpr int kRwClasses = 5;
__host__ __device__ constexpr int rw_emax(int c)
{
    return c == 0 ? 1 : c == 1 ? 3 : c == 2 ? 7 : c == 3 ? 15 : 31;
}
constexpr int kRingClasses = 3;
__host__ __device__ constexpr int ring_max_e(int c)
{
    return c == 0 ? 112 : c == 1 ? 304 : 816;
}
constexpr int kIndexClasses = 3;
__host__ __device__ constexpr int index_max_e(int c)
{
    return c == 0 ? 1664 : c == 1 ? 5920 : 10016;
}
constexpr int kCtaClasses = 3;
constexpr int kCtaThreads = 1024;
__host__ __device__ constexpr int cta_mbound(int b)
{
    return b == 0 ? 16384 : b == 1 ? 65536 : 131072;
}
constexpr int kMaxLen = 131072;  // longest pair routed for E' > 31
constexpr int kFirstRing = kRwClasses;
constexpr int kFirstIndex = kFirstRing + kRingClasses;
constexpr int kFirstCta = kFirstIndex + kIndexClasses;
constexpr int kClasses = kFirstCta + kCtaClasses;
constexpr int kLenBins = 72;
constexpr int kKeys = kClasses * kLenBins;

constexpr int kClassNone = -1;         // m == 0: answered directly
constexpr int kClassInvalid = -2;      // negative m or E
constexpr int kClassUnsupported = -3;  // too long for the staged kernels

// Effective threshold: rows beyond |s| = m-1 cannot match.
__host__ __device__ inline int eff_threshold(int m, int E)
{
    return E < m - 1 ? E : (m > 0 ? m - 1 : 0);
}

// The class of a pair for the ring teams (up to ring_limit) or the index (E'
// up to its largest).
__host__ __device__ inline int wide_class_of(
    int Ee, int ring_limit = ring_max_e(kRingClasses - 1))
{
    int c = 0;
    if (Ee <= ring_limit) {
        while (Ee > ring_max_e(c))
            ++c;
        return kFirstRing + c;
    }
    while (Ee > index_max_e(c))
        ++c;
    return kFirstIndex + c;
}

__host__ __device__ inline int class_of(int m, int E)
{
    if (m < 0 || E < 0)
        return kClassInvalid;
    if (m == 0)
        return kClassNone;
    const int Ee = eff_threshold(m, E);
    if (Ee <= 31) {
        for (int c = 0; c < kRwClasses; ++c)
            if (Ee <= rw_emax(c))
                return c;
    }
    if (m > kMaxLen)
        return kClassUnsupported;
    if (Ee <= index_max_e(kIndexClasses - 1))
        return wide_class_of(Ee);
    int b = 0;
    while (m > cta_mbound(b))
        ++b;
    return kFirstCta + b;
}

// Knobs the autotuner picks (they change speed, never results):
//   rw_max_e   -- largest E' routed thread-per-pair (15 or 31); above it a
//                 pair goes to a team (pairs per warp: 32 -> 16)
//   cw_subgrid -- columns the CTA-per-pair kernel evaluates bit-parallel
//                 across rows before the surviving runs are extended
//                 word-wise (4, 8 or 16)
struct TuneParams {
    int rw_max_e = 31;
    int cw_subgrid = 8;
    // largest E' a ring team takes (at most its classes' bound; the server's
    // passes set a smaller one)
    int ring_limit = ring_max_e(kRingClasses - 1);
};

__host__ __device__ inline int class_of_tuned(int m, int E,
                                              const TuneParams &tp)
{
    const int c = class_of(m, E), Ee = eff_threshold(m, E);
    // above the thread-per-pair limit: a team; above the teams': the index
    if (c >= 0 && c < kFirstIndex && Ee > tp.rw_max_e)
        return wide_class_of(Ee, tp.ring_limit);
    return c;
}

// The serving engine's passes: pairs above 511 edits are long ones, which
// leave their batch for the queue whose worker holds the index; in the
// batch's class kernels they would hold its slot until the last is routed.
__host__ __device__ inline TuneParams serving_params()
{
    TuneParams tp;
    tp.ring_limit = 511;
    return tp;
}

// Quarter-octave length bin, counted from the longest (bin 0) down.
__host__ __device__ inline int len_bin_desc(int m)
{
    int lb = 0;
    for (int x = m; x > 1; x >>= 1)
        ++lb;  // ceil-ish log2 is fine: only the order matters
    int fine = lb >= 2 ? ((m >> (lb - 2)) & 3) : 0;
    int bin = 4 * lb + fine;
    if (bin > kLenBins - 1)
        bin = kLenBins - 1;
    return kLenBins - 1 - bin;
}

// The batch as the kernels see it.
struct PairSet {
    const uint32_t *reads;   // packed words
    const uint32_t *refs;
    const int64_t *offsets;  // word offset per pair, or NULL (fixed stride)
    const int32_t *lengths;  // per-pair m, or NULL (uniform m)
    const int32_t *Es;       // per-pair E, or NULL (uniform e)
    int32_t m, e;
    int64_t stride;          // words per pair when offsets == NULL
    int64_t n;
    uint8_t *acc;
    int32_t *obs;
    __device__ __forceinline__ int len(int64_t p) const
    {
        return lengths ? lengths[p] : m;
    }
    __device__ __forceinline__ int thr(int64_t p) const
    {
        return Es ? Es[p] : e;
    }
    __device__ __forceinline__ int64_t off(int64_t p) const
    {
        return offsets ? offsets[p] : p * stride;
    }
};

// Workspace of the bucketing pass (device).
struct BucketWs {
    int *hist;      // kKeys
    int *ndeferred; // tiles listed in deferred (zeroed with hist)
    int *cursor;    // kKeys
    int *ranges;    // 2 * kClasses: [begin, end) per class in perm
    unsigned *counters;  // kClasses work counters of the persistent kernels
    int32_t *deferred;   // input tiles (of kRwThreads pairs) left to the classes
    int32_t *perm;  // n pair indices, grouped by key
};

// The serving engine's device-resident queue of long pairs (ss_server.cu):
// a ring of entries that producers (the enqueue kernel of each batch's
// pass) fill and a long-lived worker kernel drains.  An entry is published
// by writing its seq (= ring position + 1) last; a consumer claims position
// h by moving head from h to h + 1 only once entry h carries seq h + 1.
struct LongEntry {
    int64_t pair;
    int32_t batch;
    uint32_t seq;
};

// One batch whose long pairs are queued: where its pairs and results live.
struct LongBatch {
    PairSet ps;
    const uint8_t *bad;  // per-pair invalid-input flags (routed as -1)
    int remaining;       // queued pairs not yet routed
    int gen;             // written to done[] when remaining reaches 0
};

struct LongQueue {
    LongEntry *ring;             // kLongRing entries
    unsigned long long *tail;    // positions reserved by producers
    unsigned long long *head;    // positions claimed by consumers
    unsigned long long *last;    // time of the last claim by any worker
    int *busy;                   // worker CTAs routing a pair now
    int *closing;                // set once: every worker CTA leaves
    LongBatch *batches;          // kLongBatches descriptors
    volatile int *done;          // host-mapped: gen of each finished batch
    volatile int *stop;          // host-mapped: workers leave when set
};

constexpr int kLongRing = 1 << 18;   // entries (a power of two)
constexpr int kLongBatches = 64;     // descriptors
// Worker shape: one CTA per SM, routing a pair at a time with an index of up
// to 98 KB (a pair of 100 kbp at E = 10^4; above that all rows in 35 KB), so
// that more than half of the SM's shared memory stays free for the batches'
// own kernels (without room beside the worker they waited for it to leave).
constexpr int kLongCtasPerSm = 1;

// Whether the queue takes the pairs of class cls: the index and the CTA
// classes.  (A batch's own CTA kernel takes up to 180 KB of an SM's shared
// memory for a long pair: it would wait for the worker to leave, and hold the
// batch's slot until then.)
__host__ __device__ inline bool long_queued(int cls)
{
    return cls >= kFirstIndex;
}

// A batch's hook into the queue: its descriptor index, passed to the
// enqueue kernel of its pass.
struct LongHook {
    LongQueue q;
    int batch;
};

// Arguments of k_seg_direct (ss_seg.cu): groups of kSegGroup input tiles of
// kRwThreads pairs per CTA.
constexpr int kSegGroup = 8;
struct SegArgs {
    PairSet ps;
    BucketWs ws;
    TuneParams tp;
    int64_t ntiles;  // ceil(n / kRwThreads)
    uint32_t neg1;   // 0xffffffff (see rw_route)
    int *status;
};

}  // namespace ssk
