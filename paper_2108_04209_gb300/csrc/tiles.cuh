// Block-wide prefix sums and the prefix of tiles per problem (one CTA).
#pragma once
#include "common.cuh"

namespace {

// exclusive prefix of v over the CTA's threads, *total the sum; sh: 32 entries
template <typename T>
__device__ __forceinline__ T cta_exscan(T v, T *sh, T *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    T x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) sh[warp] = x;
    __syncthreads();
    T before = 0, all = 0;
    for (int w = 0; w < nw; w++) {
        const T s = sh[w];
        before += (w < warp) ? s : 0;
        all += s;
    }
    *total = all;
    return before + x - v;
}

// tile_off[p]: tiles of tr kept rows before problem p; tile_off[nprob] all
// (the thousand per-thread sums were added up by one thread: 7 us of a launch)
__global__ void __launch_bounds__(1024)
k_tiles(int64_t nprob, const int32_t *__restrict__ mk, int tr, int64_t *__restrict__ tile_off)
{
    __shared__ int64_t sh[32];
    const int64_t per = (nprob + blockDim.x - 1) / blockDim.x;
    const int64_t beg = min(nprob, threadIdx.x * per), end = min(nprob, beg + per);
    int64_t s = 0, all;
    for (int64_t p = beg; p < end; p++) s += (mk[p] + tr - 1) / tr;
    int64_t acc = cta_exscan(s, sh, &all);
    if (threadIdx.x == 0) tile_off[nprob] = all;
    for (int64_t p = beg; p < end; p++) { tile_off[p] = acc; acc += (mk[p] + tr - 1) / tr; }
}

// threads for k_tiles and the like: enough for one problem each, at most 1024
inline int tiles_threads(int64_t nprob) { return nprob >= 1024 ? 1024 : (int)((nprob + 31) / 32 * 32); }

}  // namespace
