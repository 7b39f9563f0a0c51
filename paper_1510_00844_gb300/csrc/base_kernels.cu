// Non-template kernels: row binning, int64 exclusive scan, empty rows; and
// their host launchers.
#include <exception>
#include <map>
#include <tuple>

#include "plan.h"

namespace sg {

__global__ void class_offsets_kernel(DevCounters* cnt, int seg_log2) {
    class_offsets(cnt, seg_log2);
}

// Scatter global row ids into their class segment (order inside a class is
// free; rows are independent).  Each block counts its rows per class in
// shared memory, reserves one range per class with a single global atomic,
// then places its rows.  Lanes of a warp with the same class are grouped, so
// one atomic per class and warp does the counting (rows of one product often
// share a class).
__global__ void bin_rows_kernel(long long R, const unsigned char* __restrict__ cls,
                                int32_t* __restrict__ rows, DevCounters* cnt) {
    __shared__ unsigned long long loc[kNumClasses];
    __shared__ unsigned long long base[kNumClasses];
    const long long per_block = (R + gridDim.x - 1) / gridDim.x;
    const long long r0 = (long long)blockIdx.x * per_block;
    const long long r1 = min(R, r0 + per_block);
    for (int t = threadIdx.x; t < kNumClasses; t += blockDim.x) loc[t] = 0;
    __syncthreads();
    bin_block_rows(cls, rows, r0, r1, loc, nullptr);
    __syncthreads();
    for (int t = threadIdx.x; t < kNumClasses; t += blockDim.x) {
        base[t] = loc[t] ? atomicAdd(&cnt->class_cursor[t], loc[t]) : 0;
        loc[t] = 0;
    }
    __syncthreads();
    bin_block_rows(cls, rows, r0, r1, loc, base);
}

// ------------------------------------------------------------------ scan
// In-place exclusive scan of int64 x[0..N).  Tiles of 4096: a warp takes 512
// consecutive entries, 16 per lane, all loaded at once (a tile taken 256
// entries at a time, with four barriers each, was 8.7 us of the 0.18 ms of a
// small product; now 3).  One tile takes one kernel, up to kScanDirect tiles
// two (every block adds up the sums of the tiles before its own), more three.
constexpr long long kScanDirect = 2048;

__global__ void __launch_bounds__(kScanThreads)
    scan_reduce_kernel(const int64_t* __restrict__ x, long long N, int64_t* __restrict__ part) {
    __shared__ long long ws[kScanThreads / 32];
    long long base = (long long)blockIdx.x * kScanTile;
    long long v[kScanItems];
#pragma unroll
    for (int t = 0; t < kScanItems; ++t) {
        const long long idx = base + (long long)t * kScanThreads + threadIdx.x;
        v[t] = idx < N ? x[idx] : 0;
    }
    long long s = 0;
#pragma unroll
    for (int t = 0; t < kScanItems; ++t) s += v[t];
    s = warp_sum(s);
    if (lane_id() == 0) ws[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        long long w = threadIdx.x < kScanThreads / 32 ? ws[threadIdx.x] : 0;
        w = warp_sum(w);
        if (threadIdx.x == 0) part[blockIdx.x] = w;
    }
}

// Exclusive scan of the tile sums with one block of 1024 threads (carry loop).
__global__ void scan_partials_kernel(int64_t* part, long long nparts) {
    __shared__ long long ws[32];
    __shared__ long long carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (long long b = 0; b < nparts; b += blockDim.x) {
        long long idx = b + threadIdx.x;
        long long v = idx < nparts ? part[idx] : 0;
        long long inc = warp_incl_scan(v);
        if (lane_id() == 31) ws[threadIdx.x >> 5] = inc;
        __syncthreads();
        if (threadIdx.x < 32) {
            long long w = ws[threadIdx.x];
            long long wi = warp_incl_scan(w);
            ws[threadIdx.x] = wi - w;
        }
        __syncthreads();
        long long excl = carry + ws[threadIdx.x >> 5] + inc - v;
        if (idx < nparts) part[idx] = excl;
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry = excl + v;
        __syncthreads();
    }
}

// part: the tiles' sums (direct), or the sums of the tiles before each.  The
// last entry's result also goes to total_out, if given.
__global__ void __launch_bounds__(kScanThreads)
    scan_apply_kernel(int64_t* __restrict__ x, long long N, const int64_t* __restrict__ part,
                      bool direct, int64_t* total_out) {
    constexpr int kWarps = kScanThreads / 32;
    __shared__ long long ws[kWarps], before[kWarps];
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const long long base = (long long)blockIdx.x * kScanTile + (long long)w * 32 * kScanItems + lane;
    long long v[kScanItems];
#pragma unroll
    for (int t = 0; t < kScanItems; ++t) v[t] = base + 32 * t < N ? x[base + 32 * t] : 0;
    long long prev = 0;
    if (direct)
        for (long long u = threadIdx.x; u < blockIdx.x; u += kScanThreads) prev += part[u];
    else if (threadIdx.x == 0)
        prev = part[blockIdx.x];
    long long s = 0;
#pragma unroll
    for (int t = 0; t < kScanItems; ++t) s += v[t];
    s = warp_sum(s);
    prev = warp_sum(prev);
    if (lane == 0) {
        ws[w] = s;
        before[w] = prev;
    }
    __syncthreads();
    long long carry = 0;
#pragma unroll
    for (int u = 0; u < kWarps; ++u) carry += before[u] + (u < w ? ws[u] : 0);
#pragma unroll
    for (int t = 0; t < kScanItems; ++t) {
        const long long incl = warp_incl_scan(v[t]);
        if (base + 32 * t < N) x[base + 32 * t] = carry + incl - v[t];
        if (total_out && base + 32 * t == N - 1) *total_out = carry + incl - v[t];
        carry += __shfl_sync(kFull, incl, 31);
    }
}

// Relative row pointers of every product: out[out_base_p + i] = g[rb_p + i] - g[rb_p].
__global__ void product_rowptr_kernel(long long R, const long long* __restrict__ rb, int nprod,
                                      const int64_t* __restrict__ g, int64_t* __restrict__ out) {
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < R + nprod;
         t += (long long)gridDim.x * blockDim.x) {
        // entry t belongs to product p with rb[p] + p <= t < rb[p+1] + p + 1
        int lo = 0, hi = nprod - 1;
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (rb[mid] + mid <= t) lo = mid;
            else hi = mid - 1;
        }
        const long long i = t - rb[lo] - lo;
        out[t] = g[rb[lo] + i] - g[rb[lo]];
    }
}

int occupancy_lookup(const void* kernel, int threads, size_t smem) {
    thread_local std::map<std::tuple<int, const void*, int, size_t>, int> known;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1;
    const auto key = std::make_tuple(dev, kernel, threads, smem);
    const auto it = known.find(key);
    if (it != known.end()) return it->second;
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, threads, smem) != cudaSuccess ||
        b < 1)
        return 1;   // an error is not remembered
    try {
        if (known.size() >= 256) known.clear();
        known[key] = b;
    } catch (const std::exception&) {   // no room to remember it
    }
    return b;
}

cudaError_t launch_class_offsets(Plan& P) {
    count_launches(1);
    class_offsets_kernel<<<1, 32, 0, P.stream>>>(P.cnt, P.seg_log2);
    return cudaGetLastError();
}

// The row analysis has formed the class offsets (there is none without rows).
cudaError_t launch_binning(Plan& P) {
    const long long R = P.R;
    if (R <= 0) return launch_class_offsets(P);
    int blocks = (int)std::max<long long>(1, std::min<long long>((R + 1023) / 1024, (long long)P.sm_count * 4));
    count_launches(1);
    bin_rows_kernel<<<blocks, 256, 0, P.stream>>>(R, P.cls, P.rows, P.cnt);
    return cudaGetLastError();
}

size_t scan_temp_bytes(long long N) {
    long long parts = (N + kScanTile - 1) / kScanTile;
    return (size_t)std::max<long long>(parts, 1) * sizeof(int64_t);
}

cudaError_t launch_exclusive_scan(int64_t* x, long long N, int64_t* temp, cudaStream_t s,
                                  int64_t* total_out) {
    if (N <= 0) return cudaSuccess;
    long long parts = (N + kScanTile - 1) / kScanTile;
    const bool direct = parts <= kScanDirect;
    if (parts > 1) {
        count_launches(1);
        scan_reduce_kernel<<<(unsigned)parts, kScanThreads, 0, s>>>(x, N, temp);
    }
    if (!direct) {
        count_launches(1);
        scan_partials_kernel<<<1, 1024, 0, s>>>(temp, parts);
    }
    count_launches(1);
    scan_apply_kernel<<<(unsigned)parts, kScanThreads, 0, s>>>(x, N, temp, direct, total_out);
    return cudaGetLastError();
}

cudaError_t launch_product_rowptr(const Plan& P, const int64_t* g, int64_t* out) {
    const long long total = P.R + P.nprod;
    int blocks = (int)std::max<long long>(1, std::min<long long>((total + 255) / 256, (long long)P.sm_count * 8));
    count_launches(1);
    product_rowptr_kernel<<<blocks, 256, 0, P.stream>>>(P.R, P.rb, P.nprod, g, out);
    return cudaGetLastError();
}

}  // namespace sg
