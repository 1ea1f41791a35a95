// ss_verify.cu -- accuracy harness kernels: capped edit distance per pair
// and the confusion counts of filter decisions against it.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "ss_internal.h"
#include "ss_pm.cuh"
#include "ss_verify.cuh"

namespace ssk {

// Pairs of one length and threshold, 32 per thread (ed_walk): 3M pairs of
// 100 bp at E = 5: 0.102 ms, where a thread per pair evaluating 2E+1 cells a
// row, ten loads each, took 3.756 ms.
template <int E>
__global__ void __launch_bounds__(kPmThreads) k_pm_ed(const PmArgs a, int32_t *ed,
                                              int vec)
{
    extern __shared__ uint32_t x[];
    PmSrc src;
    int64_t p0;
    int np;
    if (!pm_prepare(x, a, src, p0, np))
        return;
    const uint32_t pad = np >= 32 ? 0u : 0xffffffffu << np;
    SlicedCount<E> cnt;
    ed_walk<E>(src, a.m, pad, cnt);
    uint32_t cb[SlicedShape<E>::NB];
    cnt.bits(cb);
    if (np == 32 && vec) {
        uint4 *o = reinterpret_cast<uint4 *>(ed + p0);
#pragma unroll
        for (int v = 0; v < 8; ++v)
            o[v] = make_uint4((uint32_t)sliced_count<E>(cb, 4 * v),
                              (uint32_t)sliced_count<E>(cb, 4 * v + 1),
                              (uint32_t)sliced_count<E>(cb, 4 * v + 2),
                              (uint32_t)sliced_count<E>(cb, 4 * v + 3));
    } else {
        for (int i = 0; i < np; ++i)
            ed[p0 + i] = sliced_count<E>(cb, i);
    }
}

// counts[0..3] += (accepted & ED<=E, accepted & ED>E, rejected & ED<=E,
// rejected & ED>E): true accepts, false accepts, false rejects, true
// rejects (Section 3.2's rates are false accepts / (ED>E) and false
// rejects / (ED<=E)).
__global__ void k_confusion(const uint8_t *__restrict__ acc,
                            const int32_t *__restrict__ ed, int64_t n, int E,
                            unsigned long long *counts)
{
    unsigned long long c[4] = {0, 0, 0, 0};
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * blockDim.x) {
        const bool a = acc[p] != 0, close = ed[p] <= E;
        c[(a ? 0 : 2) + (close ? 0 : 1)] += 1;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        unsigned long long v = c[k];
        for (int off = 16; off > 0; off >>= 1)
            v += __shfl_down_sync(0xffffffffu, v, off);
        if ((threadIdx.x & 31) == 0 && v)
            atomicAdd(&counts[k], v);
    }
}

// Pairs of any length and threshold, TEAM lanes per pair over the diagonals
// of a step, F of the last two steps in shared memory.  The launch for
// (ELO, EHI] takes the pairs of those thresholds and skips the others; the
// first launch (ELO < 0) also flags unsupported thresholds.  The teams of a
// warp step together (a step ends when the slowest slide of the warp does).
// Bound by instruction issue: about 130 per 32 diagonals of a step, most of
// them the two window assemblies of a slide.  60,000 pairs of 64 bp to 10
// kbp, E = 5 %: 2.73 ms, where the banded table (a warp per pair, every cell
// of 2E+1 diagonals) took 111.6 ms.
struct EdVarArgs {
    const uint32_t *reads;
    const uint32_t *refs;
    const int64_t *off;   // words; NULL: pair p at word p * ceil(m/16), and
    const int32_t *len;   // bases;       every pair of m bases
    const int32_t *E;     //              at threshold e
    int32_t m, e;
    int64_t n;
    int32_t *ed;
    int *status;
};

constexpr int kEdVarWarps = 4;
// up to it 8 lanes per pair, above 32 (1.2M pairs of 250 bp at E = 16 / 31:
// 32 lanes 1989 / 2984 us, 8 lanes 994 / 2151)
constexpr int kEdTeamMaxE = 63;

template <int TEAM, int ELO, int EHI>
__global__ void __launch_bounds__(32 * kEdVarWarps)
    k_ed_diag(const EdVarArgs a)
{
    constexpr int T = 32 / TEAM;    // pairs per warp
    constexpr int H = EHI / 2;      // |k| never exceeds it
    constexpr int W = 2 * H + 3;    // and a guard entry either side
    __shared__ int s_f[kEdVarWarps][T][2][W];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int team = lane / TEAM, tl = lane % TEAM;
    int(*F)[W] = s_f[wib][team];
    const int64_t step = (int64_t)gridDim.x * kEdVarWarps * T;
    for (int64_t p0 = ((int64_t)blockIdx.x * kEdVarWarps + wib) * T;
         p0 < a.n; p0 += step) {
        const int64_t p = p0 + team;
        int m = 0, E = 0;
        bool act = p < a.n;
        if (act) {
            m = a.off ? a.len[p] : a.m;
            E = a.off ? a.E[p] : a.e;
            if (m < 0 || E < 0 || E > kEdWarpMaxE) {
                if (ELO < 0 && tl == 0) {
                    a.ed[p] = -1;
                    atomicOr(a.status, m < 0 || E < 0 ? kStatusInvalidArg
                                                      : kStatusUnsupported);
                }
                act = false;
            } else if (E <= ELO || E > EHI) {
                act = false;
            }
        }
        if (!__any_sync(0xffffffffu, act))
            continue;
        const int w16 = (m + 15) >> 4;
        const int64_t off = !act ? 0 : a.off ? a.off[p] : p * w16;
        const uint32_t *q = a.reads + off, *r = a.refs + off;
        for (int x = tl; x < W; x += TEAM)
            F[0][x] = F[1][x] = kEdNone;
        __syncwarp();
        if (act && tl == 0)
            F[0][H + 1] = ed_slide(q, r, w16, 0, 0, m);
        __syncwarp();
        for (int e = 0;; ++e) {
            if (act) {
                int ed;
                if (ed_ends(F[e & 1][H + 1], m, E, e, ed)) {
                    if (tl == 0)
                        a.ed[p] = ed;
                    act = false;
                }
            }
            if (!__any_sync(0xffffffffu, act))
                break;
            if (act)
                ed_advance(q, r, w16, m, E, e, F[e & 1] + H + 1,
                           F[(e + 1) & 1] + H + 1, tl, TEAM);
            __syncwarp();
        }
        __syncwarp();  // F is reused by the next pair
    }
}

namespace {

cudaError_t launch_diag(const EdVarArgs &a, bool small, bool large,
                        cudaStream_t st)
{
    // one warp's worth of pairs per warp (no cap on the grid: pairs differ
    // in cost by the square of their threshold, and the block scheduler
    // hands them out as warps finish)
    auto grid = [&](int teams) {
        const int64_t per = (int64_t)kEdVarWarps * teams;
        return (unsigned)std::min<int64_t>((a.n + per - 1) / per, 0x7fffffff);
    };
    if (small)
        k_ed_diag<8, -1, kEdTeamMaxE>
            <<<grid(4), 32 * kEdVarWarps, 0, st>>>(a);
    if (large)
        k_ed_diag<32, kEdTeamMaxE, kEdWarpMaxE>
            <<<grid(1), 32 * kEdVarWarps, 0, st>>>(a);
    return cudaGetLastError();
}

template <int... Es>
cudaError_t pm_ed_dispatch(int E, const PmArgs &a, int32_t *ed, unsigned grid,
                           size_t smem, cudaStream_t st,
                           std::integer_sequence<int, Es...>)
{
    const int vec = ((uintptr_t)ed & 15) == 0;
    cudaError_t r = cudaErrorInvalidValue;
    ((E == Es ? (k_pm_ed<Es><<<grid, kPmThreads, smem, st>>>(a, ed, vec),
                 r = cudaGetLastError(), 0)
              : 0),
     ...);
    return r;
}

template <int... Es>
cudaError_t pm_ed_attributes(std::integer_sequence<int, Es...>)
{
    cudaError_t r = cudaSuccess;
    ((r == cudaSuccess
          ? (r = cudaFuncSetAttribute(
                 k_pm_ed<Es>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                 kPmSmem),
             0)
          : 0),
     ...);
    return r;
}

using EdEs = std::make_integer_sequence<int, kEdMaxE + 1>;

}  // namespace

cudaError_t pm_ed_init() { return pm_ed_attributes(EdEs{}); }

// Bit-sliced or by diagonals, whichever is faster: the walk's time grows
// with the length (twice: a warp holds fewer groups), the diagonals' with
// the square of the threshold.  Measured (us, walk / diagonals): 3M pairs of
// 100 bp E = 0 83 / 638, E = 5 102 / 1002; 0.9M of 350 bp E = 0 141 / 207, E
// = 15 390 / 723; 0.6M of 500 bp E = 5 465 / 248, E = 31 1164 / 1144.  Few
// pairs leave the walk with a few lanes per warp: 33,000 of 100 bp E = 5 18
// / 26, of 250 bp E = 5 36 / 26.
static bool ed_walk_faster(int64_t n, int32_t m)
{
    const int w16 = (m + 15) / 16;
    return w16 <= 22 && n >= (w16 <= 7 ? 16384 : 65536);
}

cudaError_t launch_ed_banded(int E, const uint32_t *reads,
                             const uint32_t *refs, int64_t n, int32_t m,
                             int32_t *ed, int sm_count, cudaStream_t st)
{
    if (n <= 0)
        return cudaSuccess;
    PmArgs a;
    unsigned grid;
    size_t smem;
    if (ed_walk_faster(n, m) &&
        pm_config(reads, refs, n, m, sm_count, 0, a, grid, smem))
        return pm_ed_dispatch(E, a, ed, grid, smem, st, EdEs{});
    const EdVarArgs v{reads, refs, nullptr, nullptr, nullptr, m, E, n, ed,
                      nullptr};
    return launch_diag(v, E <= kEdTeamMaxE, E > kEdTeamMaxE, st);
}

cudaError_t launch_ed_var(const uint32_t *reads, const uint32_t *refs,
                          const int64_t *off, const int32_t *len,
                          const int32_t *E, int64_t n, int32_t *ed,
                          int *status, cudaStream_t st)
{
    if (n <= 0)
        return cudaSuccess;
    return launch_diag(
        EdVarArgs{reads, refs, off, len, E, 0, 0, n, ed, status}, true, true,
        st);
}

cudaError_t launch_confusion(const uint8_t *acc, const int32_t *ed,
                             int64_t n, int E, unsigned long long *counts,
                             int sm_count, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(counts, 0, 4 * sizeof(unsigned long long),
                                    st);
    if (e != cudaSuccess || n <= 0)
        return e;
    const int64_t want = (n + 255) / 256;
    const int grid = (int)(want < (int64_t)sm_count * 8 ? want
                                                        : (int64_t)sm_count * 8);
    k_confusion<<<grid, 256, 0, st>>>(acc, ed, n, E, counts);
    return cudaGetLastError();
}

}  // namespace ssk
