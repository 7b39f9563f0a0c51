// CSR transpose: A (m x n) -> A^T (n x m), rows of A^T with ascending column
// (= original row) indices.  The paper transposes the B blocks locally during
// redistribution (Alg. 2, the all-to-all of B); here it supplies R^T for the
// Galerkin product R^T A R.
//
// Steps, each over the entries of A in order (not over its rows, which may
// hold one entry or a hundred thousand):
//   count    every entry takes the next place of its column (atomic counter);
//   scan     of the counters = row pointers of A^T;
//   scatter  (row, value) of every entry to its place in a scratch copy of
//            A^T (arbitrary order inside a row; no further atomics);
//   sort     every row of A^T from the scratch copy into the result, by
//            original row index.  The place of an entry is the number of
//            smaller ones (and of equal ones before it in the scratch copy, for
//            an A whose rows repeat a column): rows of at most 8
//            entries take 8 lanes, of at most 32 a warp (both compare all
//            pairs in registers), of at most 256 a warp's bitonic sort in
//            shared memory; longer rows take a block and a bitmap of the
//            original rows, in which an entry's place is the set bits
//            before it, one window of the bitmap after another.
// What bounds it, in the 0.69 ms that R-MAT 18 takes (7.6 M entries): the
// scattered stores (0.26 ms, 32 sectors per store), the shared-memory sorts (0.31
// ms, L1 80 and 70 % busy) and the returning atomics (0.08 ms).  Before, one warp
// per row of A left 31 lanes idle on a restriction operator (128^3 points, one
// entry per row: count, scatter and sort 0.82 ms, now 0.1 ms) and columns
// beyond 8192 entries compared all pairs (R-MAT 18: 23.7 of 26.9 ms).
#include <cstdio>

#include "plan.h"

namespace sg {

constexpr int kTrThreads = 256;
constexpr int kTrItems = 8;                       // entries per thread
constexpr int kTrTile = kTrThreads * kTrItems;    // entries per block and step
constexpr int kTrRows = 4096;                     // row pointers held in shared memory
constexpr int kTrWarpMax = 256;                   // rows up to this take a warp
constexpr int kTrBlockMax = 8192;                 // bitonic sort in a block
constexpr int kTrWords = 14336;                   // bitmap words of a window
// Rows of at most kTrBlockMax entries take the bitmap while it has at most
// this many bits per entry (clearing and counting it then costs less than the
// block's bitonic sort).
constexpr int kTrBitsPerEntry = 2048;

// rank[p] = how many entries of p's column were counted before p; cnt[j] ends
// as the length of column j.
template <class IT>
__global__ void __launch_bounds__(kTrThreads)
    col_rank_kernel(long long m, const int64_t* __restrict__ rp, const IT* __restrict__ ci,
                    unsigned long long* __restrict__ cnt, IT* __restrict__ rank) {
    const long long p0 = rp[0], total = rp[m] - p0;
    for (long long t = (long long)blockIdx.x * kTrTile; t < total; t += (long long)gridDim.x * kTrTile) {
        long long j[kTrItems];
#pragma unroll
        for (int u = 0; u < kTrItems; ++u) {
            const long long q = t + u * kTrThreads + threadIdx.x;
            j[u] = q < total ? (long long)ci[p0 + q] : -1;
        }
        unsigned long long old[kTrItems];
#pragma unroll
        for (int u = 0; u < kTrItems; ++u) old[u] = j[u] >= 0 ? atomicAdd(&cnt[j[u]], 1ull) : 0ull;
#pragma unroll
        for (int u = 0; u < kTrItems; ++u) {
            const long long q = t + u * kTrThreads + threadIdx.x;
            if (q < total) rank[q] = (IT)old[u];
        }
    }
}

// The row of entry p: the last i in [lo, hi] with rp[i] <= p.
template <class P>
__device__ __forceinline__ long long row_of(const P* rp, long long lo, long long hi, long long p) {
    while (lo < hi) {
        const long long mid = (lo + hi + 1) >> 1;
        if (rp[mid] <= p) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

template <class IT, class V>
__global__ void __launch_bounds__(kTrThreads)
    scatter_kernel(long long m, const int64_t* __restrict__ rp, const IT* __restrict__ ci,
                   const V* __restrict__ va, const IT* __restrict__ rank,
                   const int64_t* __restrict__ rpT, IT* __restrict__ ciS, V* __restrict__ vaS) {
    __shared__ int64_t srp[kTrRows];
    __shared__ long long ends[2];
    const long long p0 = rp[0], total = rp[m] - p0;
    for (long long t = (long long)blockIdx.x * kTrTile; t < total; t += (long long)gridDim.x * kTrTile) {
        // the rows of the tile's first and last entry; the row pointers between
        // them are searched in shared memory when they fit
        if (threadIdx.x < 2) {
            const long long p = threadIdx.x == 0 ? t : min(total, t + (long long)kTrTile) - 1;
            ends[threadIdx.x] = row_of(rp, 0, m - 1, p0 + p);
        }
        __syncthreads();
        const long long r0 = ends[0], r1 = ends[1];
        const bool held = r1 - r0 < kTrRows;
        if (held)
            for (long long i = r0 + threadIdx.x; i <= r1; i += kTrThreads) srp[i - r0] = rp[i];
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kTrItems; ++u) {
            const long long q = t + u * kTrThreads + threadIdx.x;
            if (q < total) {
                const long long j = (long long)ci[p0 + q];
                const long long pos = rpT[j] + (long long)rank[q];
                V v{};
                if constexpr (VOps<V>::has_val) v = va[p0 + q];
                const long long i = held ? r0 + row_of(srp, 0, r1 - r0, p0 + q)
                                         : row_of(rp, r0, r1, p0 + q);
                ciS[pos] = (IT)i;
                if constexpr (VOps<V>::has_val) vaS[pos] = v;
            }
        }
        __syncthreads();
    }
}

// Sorts rows of at most kTrWarpMax entries from the scratch copy into the
// result and lists the longer ones.  A warp takes 32 consecutive rows.
template <class IT, class V, int WARPS>
__global__ void __launch_bounds__(WARPS * 32)
    sort_rows_kernel(long long n, const int64_t* __restrict__ rpT, const IT* __restrict__ ciS,
                     const V* __restrict__ vaS, IT* __restrict__ ciT, V* __restrict__ vaT,
                     long long* __restrict__ long_rows, unsigned* long_count) {
    constexpr bool HV = VOps<V>::has_val;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = lane_id();
    const int w = threadIdx.x >> 5;
    constexpr size_t vbytes = HV ? sizeof(V) * kTrWarpMax : 0;
    V* vals = reinterpret_cast<V*>(smem_raw + (size_t)w * (vbytes + sizeof(IT) * kTrWarpMax));
    IT* keys = reinterpret_cast<IT*>(smem_raw + (size_t)w * (vbytes + sizeof(IT) * kTrWarpMax) + vbytes);
    const IT kmax = sizeof(IT) == 4 ? (IT)0x7fffffff : (IT)0x7fffffffffffffffLL;
    const long long nw = (long long)gridDim.x * WARPS;
    for (long long tile = (long long)blockIdx.x * WARPS + w; tile * 32 < n; tile += nw) {
        const long long j = tile * 32 + lane;
        const long long a = j < n ? rpT[j] : 0;
        const long long L = j < n ? rpT[j + 1] - a : 0;
        if (L > kTrWarpMax) long_rows[atomicAdd(long_count, 1u)] = j;
        // at most 8 entries: four rows at a time
        for (unsigned small = __ballot_sync(kFull, L > 0 && L <= 8); small;) {
            // the (lane / 8)-th of the rows left
            unsigned s = small;
            for (int g = lane >> 3; g > 0 && s; --g) s &= s - 1u;
            const int src = s ? __ffs(s) - 1 : 0;
            const long long ar = __shfl_sync(kFull, a, src);
            const long long Ls = __shfl_sync(kFull, L, src);
            const int Lr = s ? (int)Ls : 0;
            const int x = lane & 7;
            const IT key = x < Lr ? ciS[ar + x] : kmax;
            V v{};
            if constexpr (HV)
                if (x < Lr) v = vaS[ar + x];
            int place = 0;
#pragma unroll
            for (int y = 0; y < 8; ++y) {
                const IT other = __shfl_sync(kFull, key, y, 8);
                place += other < key || (other == key && y < x);
            }
            if (x < Lr) {
                ciT[ar + place] = key;
                if constexpr (HV) vaT[ar + place] = v;
            }
            for (int g = 0; g < 4 && small; ++g) small &= small - 1u;
        }
        for (unsigned mid = __ballot_sync(kFull, L > 8 && L <= kTrWarpMax); mid; mid &= mid - 1u) {
            const int src = __ffs(mid) - 1;
            const long long ar = __shfl_sync(kFull, a, src);
            const int Lr = (int)__shfl_sync(kFull, L, src);
            if (Lr <= 32) {
                const IT key = lane < Lr ? ciS[ar + lane] : kmax;
                V v{};
                if constexpr (HV)
                    if (lane < Lr) v = vaS[ar + lane];
                int place = 0;
                for (int y = 0; y < Lr; ++y) {
                    const IT other = __shfl_sync(kFull, key, y);
                    place += other < key || (other == key && y < lane);
                }
                if (lane < Lr) {
                    ciT[ar + place] = key;
                    if constexpr (HV) vaT[ar + place] = v;
                }
                continue;
            }
            int N = 64;
            while (N < Lr) N <<= 1;
            for (int x = lane; x < N; x += 32) {
                keys[x] = x < Lr ? ciS[ar + x] : kmax;
                if constexpr (HV)
                    if (x < Lr) vals[x] = vaS[ar + x];
            }
            __syncwarp();
            for (int k = 2; k <= N; k <<= 1)
                for (int d = k >> 1; d > 0; d >>= 1) {
                    // pair t: the t-th index whose bit d is clear
                    for (int t = lane; t < N / 2; t += 32) {
                        const int i = 2 * t - (t & (d - 1)), o = i + d;
                        const IT ki = keys[i], ko = keys[o];
                        if ((ki > ko) == ((i & k) == 0)) {
                            keys[i] = ko;
                            keys[o] = ki;
                            if constexpr (HV) {
                                const V tv = vals[i];
                                vals[i] = vals[o];
                                vals[o] = tv;
                            }
                        }
                    }
                    __syncwarp();
                }
            for (int x = lane; x < Lr; x += 32) {
                ciT[ar + x] = keys[x];
                if constexpr (HV) vaT[ar + x] = vals[x];
            }
            __syncwarp();
        }
    }
}

// Sorts the listed rows (more than kTrWarpMax entries), one block per row.
template <class IT, class V, int THREADS>
__global__ void __launch_bounds__(THREADS)
    sort_long_rows_kernel(const long long* __restrict__ long_rows, const unsigned* long_count,
                          long long m, const int64_t* __restrict__ rpT,
                          const IT* __restrict__ ciS, const V* __restrict__ vaS,
                          IT* __restrict__ ciT, V* __restrict__ vaT) {
    constexpr bool HV = VOps<V>::has_val;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int warp_total[THREADS / 32];
    const int lane = lane_id();
    const int w = threadIdx.x >> 5;
    constexpr int nwarps = THREADS / 32;
    uint2* map = reinterpret_cast<uint2*>(smem_raw);   // {bits, set bits before the word}
    const long long nitems = (long long)*long_count;
    for (long long it = blockIdx.x; it < nitems; it += gridDim.x) {
        const long long j = long_rows[it];
        const long long a = rpT[j];
        const long long L = rpT[j + 1] - a;
        if (L <= kTrBlockMax && m > (long long)kTrBitsPerEntry * L) {
            // sparse row of a tall matrix: bitonic sort of (row, place) pairs
            long long* keys = reinterpret_cast<long long*>(smem_raw);
            unsigned short* from = reinterpret_cast<unsigned short*>(keys + kTrBlockMax);
            int N = 512;
            while (N < L) N <<= 1;
            for (int x = threadIdx.x; x < N; x += THREADS) {
                keys[x] = x < L ? (long long)ciS[a + x] : 0x7fffffffffffffffLL;
                from[x] = (unsigned short)x;
            }
            __syncthreads();
            for (int k = 2; k <= N; k <<= 1)
                for (int d = k >> 1; d > 0; d >>= 1) {
                    for (int t = threadIdx.x; t < N / 2; t += THREADS) {
                        const int i = 2 * t - (t & (d - 1)), o = i + d;
                        const long long ki = keys[i], ko = keys[o];
                        if ((ki > ko) == ((i & k) == 0)) {
                            keys[i] = ko;
                            keys[o] = ki;
                            const unsigned short f = from[i];
                            from[i] = from[o];
                            from[o] = f;
                        }
                    }
                    __syncthreads();
                }
            for (int x = threadIdx.x; x < L; x += THREADS) {
                ciT[a + x] = (IT)keys[x];
                if constexpr (HV) vaT[a + x] = vaS[a + from[x]];
            }
            __syncthreads();
            continue;
        }
        long long done = 0;   // entries of earlier windows
        for (long long r0 = 0; r0 < m; r0 += 32LL * kTrWords) {
            const int nwords = (int)min((long long)kTrWords, (m - r0 + 31) >> 5);
            for (int t = threadIdx.x; t < nwords; t += THREADS) map[t] = make_uint2(0u, 0u);
            __syncthreads();
            for (long long x = threadIdx.x; x < L; x += THREADS) {
                const long long d = (long long)ciS[a + x] - r0;
                if (d >= 0 && d < 32LL * nwords) atomicOr(&map[d >> 5].x, 1u << (d & 31));
            }
            __syncthreads();
            // set bits before every word: warp w owns words [t0, t1)
            const int per = ((nwords + nwarps - 1) / nwarps + 31) & ~31;
            const int t0 = min(nwords, w * per), t1 = min(nwords, t0 + per);
            int part = 0;
            for (int t = t0 + lane; t < t1; t += 32) part += __popc(map[t].x);
            part = warp_sum(part);
            if (lane == 0) warp_total[w] = part;
            __syncthreads();
            const int all = lane < nwarps ? warp_total[lane] : 0;
            int before = warp_sum(lane < w ? all : 0);
            const int total = warp_sum(all);
            for (int t = t0; t < t1; t += 32) {
                const int pc = t + lane < t1 ? __popc(map[t + lane].x) : 0;
                const int incl = warp_incl_scan(pc);
                if (t + lane < t1) map[t + lane].y = (unsigned)(before + incl - pc);
                before += __shfl_sync(kFull, incl, 31);
            }
            __syncthreads();
            for (long long x = threadIdx.x; x < L; x += THREADS) {
                const IT key = ciS[a + x];
                const long long d = (long long)key - r0;
                if (d >= 0 && d < 32LL * nwords) {
                    const uint2 e = map[d >> 5];
                    const long long pos = a + done + e.y + __popc(e.x & ((1u << (d & 31)) - 1u));
                    ciT[pos] = key;
                    if constexpr (HV) vaT[pos] = vaS[a + x];
                }
            }
            __syncthreads();
            done += total;
        }
        if (done < L) {
            // fewer rows than entries: a column is repeated in a row of A, and the
            // bitmap holds one of the two.  Every entry counts those before it
            for (long long x = threadIdx.x; x < L; x += THREADS) {
                const IT key = ciS[a + x];
                long long place = 0;
                for (long long y = 0; y < L; ++y) {
                    const IT other = ciS[a + y];
                    place += other < key || (other == key && y < x);
                }
                ciT[a + place] = key;
                if constexpr (HV) vaT[a + place] = vaS[a + x];
            }
            __syncthreads();
        }
    }
}

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

template <class IT, class V>
cudaError_t launch_transpose(const spgemm_csr& A, cudaStream_t s, unsigned char* ws,
                             int64_t* rpT, void* ciT_, void* vaT_) {
    const long long m = A.nrows, n = A.ncols, nnz = A.nnz;
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    IT* ciT = (IT*)ciT_;
    V* vaT = (V*)vaT_;
    constexpr size_t vsz = VOps<V>::has_val ? sizeof(V) : 0;
    int64_t* temp = (int64_t*)ws;
    IT* ciS = (IT*)(ws + align256(scan_temp_bytes(n + 1)));
    V* vaS = (V*)((unsigned char*)ciS + align256((size_t)nnz * sizeof(IT)));
    unsigned* long_count = (unsigned*)((unsigned char*)vaS + align256((size_t)nnz * vsz));
    long long* long_rows = (long long*)((unsigned char*)long_count + 256);
    cudaError_t e;
    if ((e = cudaMemsetAsync(rpT, 0, (size_t)(n + 1) * sizeof(int64_t), s)) != cudaSuccess) return e;
    auto blocks = [&](long long items, int per, int most) {
        return (unsigned)std::max<long long>(1, std::min<long long>((items + per - 1) / per, (long long)sms * most));
    };
    const bool entries = m > 0 && n > 0 && nnz > 0;
    if (entries) {
        // the ranks wait in the result's column array until the rows are sorted into it
        count_launches(1);
        col_rank_kernel<IT><<<blocks(nnz, kTrTile, 8), kTrThreads, 0, s>>>(
            m, A.rowptr, (const IT*)A.col, (unsigned long long*)rpT, ciT);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if ((e = launch_exclusive_scan(rpT, n + 1, temp, s)) != cudaSuccess) return e;
    if (!entries) return cudaSuccess;
    if ((e = cudaMemsetAsync(long_count, 0, sizeof(unsigned), s)) != cudaSuccess) return e;
    count_launches(3);
    scatter_kernel<IT, V><<<blocks(nnz, kTrTile, 8), kTrThreads, 0, s>>>(
        m, A.rowptr, (const IT*)A.col, (const V*)A.val, ciT, rpT, ciS, vaS);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    {
        constexpr int WARPS = 8;
        const size_t smem = (size_t)WARPS * kTrWarpMax * (sizeof(IT) + vsz);   // at most 32 KB
        sort_rows_kernel<IT, V, WARPS><<<blocks(n, 32 * WARPS, 6), WARPS * 32, smem, s>>>(
            n, rpT, ciS, vaS, ciT, vaT, long_rows, long_count);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    {
        constexpr int THREADS = 512;
        auto k = sort_long_rows_kernel<IT, V, THREADS>;
        const size_t bitonic = (size_t)kTrBlockMax * (sizeof(long long) + sizeof(unsigned short));
        const size_t bitmap = sizeof(uint2) * (size_t)std::min<long long>(kTrWords, (m + 31) / 32);
        // a row that takes the bitonic sort has m > kTrBitsPerEntry * kTrWarpMax
        const size_t smem = m > (long long)kTrBitsPerEntry * kTrWarpMax ? std::max(bitonic, bitmap) : bitmap;
        // the limit belongs to the kernel: a call of another height, in another
        // thread, must find the same one
        const size_t most = std::max(bitonic, sizeof(uint2) * (size_t)kTrWords);
        if (smem > 48 * 1024 &&
            (e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most)) != cudaSuccess)
            return e;
        k<<<blocks(std::min<long long>(n, nnz / kTrWarpMax + 1), 1, smem > 74 * 1024 ? 2 : 3), THREADS, smem, s>>>(
            long_rows, long_count, m, rpT, ciS, vaS, ciT, vaT);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace sg

extern "C" {

size_t spgemm_transpose_workspace_size(const spgemm_csr* A) {
    if (!A) return 0;
    const size_t n = (size_t)std::max<long long>(0, A->ncols);
    const size_t nnz = (size_t)std::max<long long>(0, A->nnz);
    const size_t isz = A->index_type == SPGEMM_INDEX_I32 ? 4 : 8;
    const size_t vsz = A->value_type == SPGEMM_F32 ? 4 : A->value_type == SPGEMM_BOOL ? 0 : 8;
    return sg::align256(sg::scan_temp_bytes((long long)n + 1)) + sg::align256(nnz * isz) +
           sg::align256(nnz * vsz) + 256 + sg::align256((nnz / sg::kTrWarpMax + 1) * 8);
}

spgemm_status spgemm_transpose(const spgemm_csr* A, void* stream, void* ws, size_t ws_bytes,
                               int64_t* rowptrT, void* colT, void* valT) {
    sg::set_last_error("");
    if (!A || !rowptrT || (A->nnz > 0 && !colT)) {
        sg::set_last_error("NULL argument");
        return SPGEMM_ERR_INVALID_ARG;
    }
    if (A->rowend || A->nrows < 0 || A->ncols < 0 || A->nnz < 0 || !A->rowptr ||
        (A->nnz > 0 && !A->col)) {
        sg::set_last_error("A must be a plain CSR with non-negative sizes");
        return SPGEMM_ERR_INVALID_ARG;
    }
    const bool has_val = A->value_type != SPGEMM_BOOL;
    if (has_val && A->nnz > 0 && (!A->val || !valT)) {
        sg::set_last_error("values are NULL");
        return SPGEMM_ERR_INVALID_ARG;
    }
    if (A->index_type == SPGEMM_INDEX_I32 && A->nrows > 0x7fffffffLL) {
        sg::set_last_error("rows of A exceed int32 column indices of A^T");
        return SPGEMM_ERR_INDEX_OVERFLOW;
    }
    if (!ws || ws_bytes < spgemm_transpose_workspace_size(A) || ((uintptr_t)ws) % 256) {
        sg::set_last_error("transpose workspace missing, too small or not 256-byte aligned");
        return SPGEMM_ERR_OUT_OF_MEMORY;
    }
    cudaStream_t s = (cudaStream_t)stream;
    unsigned char* w = (unsigned char*)ws;
    const bool i32 = A->index_type == SPGEMM_INDEX_I32;
    cudaError_t e;
    switch (A->value_type) {
        case SPGEMM_F64:
            e = i32 ? sg::launch_transpose<int32_t, double>(*A, s, w, rowptrT, colT, valT)
                    : sg::launch_transpose<int64_t, double>(*A, s, w, rowptrT, colT, valT);
            break;
        case SPGEMM_F32:
            e = i32 ? sg::launch_transpose<int32_t, float>(*A, s, w, rowptrT, colT, valT)
                    : sg::launch_transpose<int64_t, float>(*A, s, w, rowptrT, colT, valT);
            break;
        case SPGEMM_I64:
            e = i32 ? sg::launch_transpose<int32_t, int64_t>(*A, s, w, rowptrT, colT, valT)
                    : sg::launch_transpose<int64_t, int64_t>(*A, s, w, rowptrT, colT, valT);
            break;
        default:
            e = i32 ? sg::launch_transpose<int32_t, sg::NoVal>(*A, s, w, rowptrT, colT, nullptr)
                    : sg::launch_transpose<int64_t, sg::NoVal>(*A, s, w, rowptrT, colT, nullptr);
            break;
    }
    if (e != cudaSuccess) {
        char buf[256];
        snprintf(buf, sizeof(buf), "transpose: CUDA error %d (%s)", (int)e, cudaGetErrorString(e));
        sg::set_last_error(buf);
        return SPGEMM_ERR_CUDA;
    }
    return SPGEMM_OK;
}

}  // extern "C"
