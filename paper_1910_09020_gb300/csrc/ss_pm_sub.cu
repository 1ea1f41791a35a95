// ss_pm_sub.cu -- the sub-maze mode (Section 2.5) over pair-major packed
// pairs walked bit-sliced (ss_pm.cuh): the walk with every row restarting at
// each sub-maze's first column and at most y counted segments per sub-maze.
#include <cuda_runtime.h>

#include <cstdint>
#include <utility>

#include "ss_device.cuh"
#include "ss_internal.h"
#include "ss_pm.cuh"
#include "ss_sliced.cuh"

namespace ssk {

namespace {

struct PmSubArgs {
    PmArgs b;
    uint8_t *acc;
    int32_t *obs;
    int32_t vec;   // acc and obs 16-byte aligned
    int32_t t, y;  // sub-maze width and segments counted
};

template <int E>
__global__ void __launch_bounds__(kPmThreads) k_pm_submaze(const PmSubArgs a)
{
    extern __shared__ uint32_t x[];
    __shared__ uint32_t vtab[SlicedEdges<E>::kRows * SlicedShape<E>::WW];
    constexpr int WW = SlicedShape<E>::WW;
    const SlicedEdges<E> ed(a.b.m);
    for (int i = threadIdx.x; i < ed.rows() * WW; i += kPmThreads)
        vtab[i] = SlicedEdges<E>::valid(ed.block_of(i / WW), i % WW, a.b.m);
    PmSrc src;
    int64_t p0;
    int np;
    if (!pm_prepare(x, a.b, src, p0, np))  // (synchronises the warp)
        return;
    const uint32_t pad = np >= 32 ? 0u : 0xffffffffu << np;
    SlicedCount<E> cnt;
    sliced_walk<E>(src, a.b.m, pad, cnt, vtab, a.b.one,
                   SlicedSubMaze<E>(a.t, a.y));
    sliced_store<E>(cnt, a.acc, a.obs, p0, np, a.vec != 0);
}

template <int... I>
cudaError_t pm_dispatch(int E, const PmSubArgs &a, unsigned grid,
                        size_t smem, cudaStream_t st,
                        std::integer_sequence<int, I...>)
{
    cudaError_t r = cudaErrorInvalidValue;
    ((E == I ? (k_pm_submaze<I><<<grid, kPmThreads, smem, st>>>(a),
                r = cudaGetLastError(), 0)
             : 0),
     ...);
    return r;
}

template <int... I>
cudaError_t pm_attributes(std::integer_sequence<int, I...>)
{
    cudaError_t r = cudaSuccess;
    ((r == cudaSuccess
          ? (r = cudaFuncSetAttribute(
                 k_pm_submaze<I>,
                 cudaFuncAttributeMaxDynamicSharedMemorySize, kPmSmem),
             0)
          : 0),
     ...);
    return r;
}

using AllE = std::make_integer_sequence<int, kSlicedMaxE + 1>;

}  // namespace

cudaError_t pm_submaze_init() { return pm_attributes(AllE{}); }

// Against a thread per pair (k_submaze_pipe), t = 8, y = 3, in us (thread ->
// walk), 3M pairs of 100 bp; 2M of 150; 1.2M of 250: E = 0 92 -> 96; 84 ->
// 113; 98 -> 144, E = 5 244 -> 127; 227 -> 160; 223 -> 232, E = 10 269 ->
// 151; 239 -> 254; 240 -> 288, E = 20 1314 -> 229; 1077 -> 268; 999 -> 399.
// A warp holds fewer groups the longer the pairs, and the thread per pair
// has no column walk above E = 15.
bool pm_submaze_faster(int32_t m, int32_t E)
{
    const int w16 = (m + 15) / 16;
    return E >= 1 && E <= kSlicedMaxE &&
           w16 <= (E <= 7 ? 10 : E <= 15 ? 7 : 16);
}

cudaError_t launch_pm_submaze(const uint32_t *reads, const uint32_t *refs,
                              int64_t n, int32_t m, int32_t E, int32_t t,
                              int32_t y, uint8_t *acc, int32_t *obs,
                              int sm_count, cudaStream_t st)
{
    PmSubArgs a;
    unsigned grid;
    size_t smem;
    if (E < 0 || E > kSlicedMaxE)
        return cudaErrorInvalidValue;
    // the edge blocks' table of the threshold
    const size_t nbh = (size_t)(E + 3) / 4;
    const size_t fixed = (2 * nbh + 2) * 4 * (2 * nbh + 1) * 4;
    if (!pm_config(reads, refs, n, m, sm_count, fixed, a.b, grid, smem))
        return cudaErrorInvalidValue;
    a.acc = acc;
    a.obs = obs;
    a.vec = ((((uintptr_t)acc) | ((uintptr_t)obs)) & 15) == 0;
    a.t = t;
    a.y = y;
    return pm_dispatch(E, a, grid, smem, st, AllE{});
}

}  // namespace ssk
