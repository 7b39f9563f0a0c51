// Markov-clustering epilogue on the expansion product (the paper squares
// matrices to represent MCL expansion, Sec. 5.3): on M^T stored in CSR (rows
// of M^T are the columns of M), drop every entry below `threshold` and divide
// each row by the sum of its kept entries, so M stays column-stochastic.
// Input may be a view (rowend); output is a plain CSR of float64 values.
// Pass 1: kept count and kept sum per row; scan; pass 2: the kept entries, in
// order, divided by the row sum.  A row's sum is formed in an order that its
// length alone fixes (a warp's lanes side by side, or a block's threads for a
// row of more than kMclLong entries), so results repeat exactly from run to
// run and do not depend on how the row is stored.
// What bounds it: the FP64 pipe, which a warp's compare, add or (ten
// instructions) division takes however many lanes are active.  So values are
// compared as integers, and divided after they have been compacted, 32 at a
// time.  R-MAT, 40009 vertices (87 M entries, rows up to 23467): count 0.51 ->
// 0.31 ms, fill 2.33 -> 0.80 ms (a warp per row, one load in flight per lane, and
// divisions where the kept entries stood).
#include <cstdio>

#include "plan.h"
#include "rows.cuh"

namespace sg {

constexpr long long kMclLong = 2048;

// v >= threshold without the FP64 pipe: for a positive threshold the bits of
// doubles compare like integers (negative values below, NaN above infinity).
struct AtLeast {
    double threshold;
    __device__ __forceinline__ bool operator()(double v) const {
        if (__double_as_longlong(threshold) > 0) {
            const long long b = __double_as_longlong(v);
            return b >= __double_as_longlong(threshold) && b <= 0x7ff0000000000000LL;
        }
        return v >= threshold;
    }
};

__global__ void __launch_bounds__(kRowWarps * 32)
    mcl_count_kernel(long long m, const int64_t* __restrict__ rp, const int64_t* __restrict__ re,
                     const double* __restrict__ val, double thr, int64_t* __restrict__ cnt,
                     double* __restrict__ sums) {
    const AtLeast keeps{thr};
    __shared__ long long part_c[kRowWarps];
    __shared__ double part_s[kRowWarps];
    for_rows(
        m, kMclLong, [&](long long i) { return (re ? re[i] : rp[i + 1]) - rp[i]; },
        [&](long long i, int w, auto warps) {
            constexpr int WARPS = decltype(warps)::value;
            constexpr int stride = 32 * WARPS;
            const long long a = rp[i], b = re ? re[i] : rp[i + 1];
            long long c = 0;
            double s = 0.0;
            for (long long q0 = a + 32 * w + lane_id(); q0 < b; q0 += 4 * stride) {
                double v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = q0 + u * stride < b ? val[q0 + u * stride] : 0.0;
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (q0 + u * stride < b && keeps(v[u])) {
                        ++c;
                        s = __dadd_rn(s, v[u]);
                    }
            }
            c = warp_sum(c);
#pragma unroll
            for (int d = 16; d; d >>= 1) s = __dadd_rn(s, __shfl_xor_sync(kFull, s, d));
            if constexpr (WARPS > 1) {
                if (lane_id() == 0) {
                    part_c[w] = c;
                    part_s[w] = s;
                }
                __syncthreads();
                c = 0;
                s = 0.0;
                for (int t = 0; t < WARPS; ++t) {
                    c += part_c[t];
                    s = __dadd_rn(s, part_s[t]);
                }
            }
            if (w == 0 && lane_id() == 0) {
                cnt[i] = c;
                sums[i] = s;
            }
        });
}

template <class IT>
__global__ void __launch_bounds__(kRowWarps * 32)
    mcl_fill_kernel(long long m, const int64_t* __restrict__ rp, const int64_t* __restrict__ re,
                    const IT* __restrict__ col, const double* __restrict__ val, double thr,
                    const double* __restrict__ sums, const int64_t* __restrict__ rpo,
                    IT* __restrict__ colo, double* valo) {
    const AtLeast keeps{thr};
    for_rows(
        m, kMclLong, [&](long long i) { return (re ? re[i] : rp[i + 1]) - rp[i]; },
        [&](long long i, int w, auto warps) {
            const long long a = rp[i], n = (re ? re[i] : rp[i + 1]) - a, out = rpo[i];
            const double s = sums[i];
            constexpr int WARPS = decltype(warps)::value;
            constexpr int wide = 32 * WARPS;
            double v[4];
            long long at[4];
            filter_entries<WARPS>(
                n, w,
                [&](long long q, int stride) {
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        at[u] = a + q + u * stride;
                        v[u] = q + u * stride < n ? val[at[u]] : 0.0;
                    }
                },
                [&](int u) { return keeps(v[u]); },
                [&](int u, long long pos) {
                    colo[out + pos] = col[at[u]];
                    valo[out + pos] = v[u];
                });
            if constexpr (WARPS > 1) __syncthreads();
            else __syncwarp();
            // the row's kept values, now side by side
            const long long end = rpo[i + 1];
            for (long long q = out + 32 * w + lane_id(); q < end; q += 4 * wide) {
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = q + u * wide < end ? valo[q + u * wide] : 1.0;
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (q + u * wide < end) valo[q + u * wide] = __ddiv_rn(v[u], s);
            }
        });
}

}  // namespace sg

namespace {

spgemm_status mfail(spgemm_status st, const char* msg) {
    sg::set_last_error(msg);
    return st;
}

spgemm_status mcheck(const spgemm_csr* C) {
    if (!C || !C->rowptr || C->nrows < 0 || (C->nnz > 0 && (!C->col || !C->val)))
        return mfail(SPGEMM_ERR_INVALID_ARG, "mcl: NULL or malformed matrix");
    if (C->value_type != SPGEMM_F64) return mfail(SPGEMM_ERR_NOT_SUPPORTED, "mcl: float64 values only");
    return SPGEMM_OK;
}

size_t al(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace

extern "C" {

size_t spgemm_mcl_workspace_size(int64_t m) {
    if (m < 0) m = 0;
    return al((size_t)m * 8) + al(sg::scan_temp_bytes(m + 1));
}

spgemm_status spgemm_mcl_prune_count(const spgemm_csr* C, double threshold, void* stream,
                                     void* ws, size_t ws_bytes, int64_t* rowptrP,
                                     int64_t* nnz_host) {
    sg::set_last_error("");
    spgemm_status st = mcheck(C);
    if (st != SPGEMM_OK) return st;
    const long long m = C->nrows;
    if (!rowptrP || !nnz_host || !ws || ws_bytes < spgemm_mcl_workspace_size(m))
        return mfail(SPGEMM_ERR_INVALID_ARG, "mcl: outputs or workspace missing");
    cudaStream_t s = (cudaStream_t)stream;
    double* sums = (double*)ws;
    int64_t* temp = (int64_t*)((unsigned char*)ws + al((size_t)m * 8));
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = cudaMemsetAsync(rowptrP + m, 0, 8, s);
    if (e == cudaSuccess && m > 0) {
        const unsigned g = (unsigned)std::max<long long>(1, std::min<long long>((m + 7) / 8, (long long)sms * 8));
        sg::count_launches(1);
        sg::mcl_count_kernel<<<g, sg::kRowWarps * 32, 0, s>>>(m, C->rowptr, C->rowend,
                                                              (const double*)C->val, threshold,
                                                              rowptrP, sums);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = sg::launch_exclusive_scan(rowptrP, m + 1, temp, s);
    int64_t total = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&total, rowptrP + m, 8, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return mfail(SPGEMM_ERR_CUDA, cudaGetErrorString(e));
    *nnz_host = total;
    return SPGEMM_OK;
}

spgemm_status spgemm_mcl_prune_fill(const spgemm_csr* C, double threshold, void* stream, void* ws,
                                    size_t ws_bytes, const int64_t* rowptrP, void* colP,
                                    double* valP) {
    sg::set_last_error("");
    spgemm_status st = mcheck(C);
    if (st != SPGEMM_OK) return st;
    const long long m = C->nrows;
    if (!rowptrP || !ws || ws_bytes < spgemm_mcl_workspace_size(m))
        return mfail(SPGEMM_ERR_INVALID_ARG, "mcl: outputs or workspace missing");
    if (m == 0) return SPGEMM_OK;
    cudaStream_t s = (cudaStream_t)stream;
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const unsigned g = (unsigned)std::max<long long>(1, std::min<long long>((m + 7) / 8, (long long)sms * 8));
    sg::count_launches(1);
    if (C->index_type == SPGEMM_INDEX_I32)
        sg::mcl_fill_kernel<int32_t><<<g, sg::kRowWarps * 32, 0, s>>>(m, C->rowptr, C->rowend, (const int32_t*)C->col,
                                                       (const double*)C->val, threshold, (const double*)ws,
                                                       rowptrP, (int32_t*)colP, valP);
    else
        sg::mcl_fill_kernel<int64_t><<<g, sg::kRowWarps * 32, 0, s>>>(m, C->rowptr, C->rowend, (const int64_t*)C->col,
                                                       (const double*)C->val, threshold, (const double*)ws,
                                                       rowptrP, (int64_t*)colP, valP);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return mfail(SPGEMM_ERR_CUDA, cudaGetErrorString(e));
    return SPGEMM_OK;
}

}  // extern "C"
