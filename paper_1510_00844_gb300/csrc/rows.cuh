// Row loops of the kernels that filter or copy the rows of a finished matrix
// (masks, the Markov epilogue, compaction).  A block of eight warps takes eight
// rows at a time: a warp per row, and the whole block for a row longer than
// `limit` (one warp would walk a power-law graph's longest row alone while
// the rest of the GPU has finished).
#pragma once

#include "device_common.cuh"

namespace sg {

constexpr int kRowWarps = 8;

// f(row, warp, warps): warp w of `warps` (1 or kRowWarps) takes part in `row`;
// with kRowWarps every thread of the block does, and f may use __syncthreads.
template <class Len, class F>
__device__ __forceinline__ void for_rows(long long m, long long limit, Len&& len, F&& f) {
    __shared__ int is_long[kRowWarps];
    const int w = threadIdx.x >> 5;
    for (long long tile = blockIdx.x; tile * kRowWarps < m; tile += gridDim.x) {
        const long long i = tile * kRowWarps + w;
        const bool big = i < m && len(i) > limit;
        if (lane_id() == 0) is_long[w] = big;
        if (i < m && !big) f(i, 0, std::integral_constant<int, 1>{});
        if (!__syncthreads_or(big)) continue;
        // every flag is read before the first barrier below, so that no warp
        // sees the next tile's
        unsigned longs = 0u;
        for (int r = 0; r < kRowWarps; ++r) longs |= is_long[r] ? 1u << r : 0u;
        for (int r = 0; r < kRowWarps; ++r)
            if ((longs >> r) & 1u) {
                f(tile * kRowWarps + r, w, std::integral_constant<int, kRowWarps>{});
                __syncthreads();
            }
    }
}

// Walks entries [0, n) in steps of 4 x 32 x WARPS: load(x0, stride) takes the
// entries x0 + u * stride (u = 0..3) of this lane, keep(u) says whether the
// u-th stays and put(u, pos) writes it to place pos; places follow the
// order of the entries.
template <int WARPS, class Load, class Keep, class Put>
__device__ __forceinline__ void filter_entries(long long n, int w, Load&& load, Keep&& keep,
                                               Put&& put) {
    __shared__ int part[2][4 * kRowWarps];
    constexpr int stride = 32 * WARPS;
    long long done = 0;
    int flip = 0;
    for (long long x = 32 * w + lane_id(); x - lane_id() - 32 * w < n; x += 4 * stride) {
        load(x, stride);
        unsigned have[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) have[u] = __ballot_sync(kFull, x + u * stride < n && keep(u));
        int before[4];   // kept entries before this warp's in group u
        int total = 0;
        if constexpr (WARPS == 1) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                before[u] = total;
                total += __popc(have[u]);
            }
        } else {
            // group u of warp w is part u * WARPS + w
            static_assert(4 * WARPS == 32, "a lane per part");
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (lane_id() == 0) part[flip][u * WARPS + w] = __popc(have[u]);
            __syncthreads();
            const int v = part[flip][lane_id()];
            const int incl = warp_incl_scan(v);
            total = __shfl_sync(kFull, incl, 31);
#pragma unroll
            for (int u = 0; u < 4; ++u) before[u] = __shfl_sync(kFull, incl - v, u * WARPS + w);
            flip ^= 1;   // the next step's parts go elsewhere: one barrier per step
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if ((have[u] >> lane_id()) & 1u)
                put(u, done + before[u] + __popc(have[u] & lanemask_lt()));
        done += total;
    }
}

// at[u] = first place in the ascending col[0..n) whose column is not below
// j[u] (four searches in step, their loads in flight together).
template <class IT>
__device__ __forceinline__ void lower_bound4(const IT* __restrict__ col, long long n,
                                             const IT (&j)[4], long long (&at)[4]) {
#pragma unroll
    for (int u = 0; u < 4; ++u) at[u] = 0;
    if (n <= 0) return;
    for (long long len = n; len > 1;) {
        const long long half = len >> 1;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (col[at[u] + half - 1] < j[u]) at[u] += half;
        len -= half;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (col[at[u]] < j[u]) ++at[u];
}

}  // namespace sg
