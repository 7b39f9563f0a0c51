// Masked product (the structural mask that MIS-2 aggregation applies to its
// semiring products, Alg. 3): keep the entries of C whose (i, j) is in the
// pattern of M (complement = 0) or not in it (complement = 1).  The mask is
// applied to the rows of the finished product: the entries of the shorter of
// C(i,:) and M(i,:) are looked up in the other by binary search (for the
// complement's entries themselves C(i,:) is walked); pass 1 counts the kept
// entries, a scan gives the row pointers, pass 2 copies them in order.  The
// product's own work is not reduced by the mask.
// What bounds it: the latency of the searches, and of the longest search at a
// block's barrier (issue 12 %, DRAM 14 %).  A mask's rows are mostly far
// shorter than the product's (R-MAT, 30011 vertices, A inside A.A: 0.75 M
// entries of M against 99 M of C): looking up every entry of C, a warp per
// row, took 1.65 ms to count and 2.08 ms to fill; this takes 0.25 and 0.19.
#include <cstdio>

#include "plan.h"
#include "rows.cuh"

namespace sg {

// Rows whose walked list is longer than this take a block.
constexpr long long kMaskLong = 512;

template <class IT>
struct MaskRow {
    const IT* c;
    const IT* m;
    long long nc, nm;
};

template <class IT>
__device__ __forceinline__ MaskRow<IT> mask_row(long long i, const int64_t* rp, const int64_t* re,
                                                const IT* col, const int64_t* mrp,
                                                const int64_t* mre, const IT* mcol) {
    const long long a = rp[i], b = re ? re[i] : rp[i + 1];
    const long long ma = mrp[i], mb = mre ? mre[i] : mrp[i + 1];
    return MaskRow<IT>{col + a, mcol + ma, b - a, mb - ma};
}

template <class IT>
__global__ void __launch_bounds__(kRowWarps * 32)
    mask_count_kernel(long long m, const int64_t* __restrict__ rp, const int64_t* __restrict__ re,
                      const IT* __restrict__ col, const int64_t* __restrict__ mrp,
                      const int64_t* __restrict__ mre, const IT* __restrict__ mcol, int complement,
                      int64_t* __restrict__ cnt) {
    __shared__ long long sum;
    for_rows(
        m, kMaskLong,
        [&](long long i) {
            const MaskRow<IT> r = mask_row<IT>(i, rp, re, col, mrp, mre, mcol);
            return min(r.nc, r.nm);
        },
        [&](long long i, int w, auto warps) {
            constexpr int WARPS = decltype(warps)::value;
            const MaskRow<IT> r = mask_row<IT>(i, rp, re, col, mrp, mre, mcol);
            const bool by_mask = r.nm <= r.nc;
            const IT* x = by_mask ? r.m : r.c;
            const IT* y = by_mask ? r.c : r.m;
            const long long nx = by_mask ? r.nm : r.nc, ny = by_mask ? r.nc : r.nm;
            int both = 0;
            for (long long q0 = 32 * w; q0 < nx; q0 += 128 * WARPS) {
                IT j[4];
                long long at[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const long long q = q0 + u * 32 * WARPS + lane_id();
                    j[u] = q < nx ? x[q] : IT(-1);   // no column is negative
                }
                lower_bound4<IT>(y, ny, j, at);
#pragma unroll
                for (int u = 0; u < 4; ++u) both += at[u] < ny && y[at[u]] == j[u];
            }
            both = warp_sum(both);
            long long total = both;
            if constexpr (WARPS > 1) {
                if (threadIdx.x == 0) sum = 0;
                __syncthreads();
                if (lane_id() == 0) atomicAdd((unsigned long long*)&sum, (unsigned long long)both);
                __syncthreads();
                total = sum;
            }
            if (w == 0 && lane_id() == 0) cnt[i] = complement ? r.nc - total : total;
        });
}

template <class IT, class V>
__global__ void __launch_bounds__(kRowWarps * 32)
    mask_fill_kernel(long long m, const int64_t* __restrict__ rp, const int64_t* __restrict__ re,
                     const IT* __restrict__ col, const V* __restrict__ val,
                     const int64_t* __restrict__ mrp, const int64_t* __restrict__ mre,
                     const IT* __restrict__ mcol, int complement,
                     const int64_t* __restrict__ rpo, IT* __restrict__ colo,
                     V* __restrict__ valo) {
    constexpr bool HV = VOps<V>::has_val;
    for_rows(
        m, kMaskLong,
        [&](long long i) {
            const MaskRow<IT> r = mask_row<IT>(i, rp, re, col, mrp, mre, mcol);
            return complement ? r.nc : min(r.nc, r.nm);
        },
        [&](long long i, int w, auto warps) {
            constexpr int WARPS = decltype(warps)::value;
            const MaskRow<IT> r = mask_row<IT>(i, rp, re, col, mrp, mre, mcol);
            const bool by_mask = !complement && r.nm <= r.nc;
            const IT* x = by_mask ? r.m : r.c;
            const IT* y = by_mask ? r.c : r.m;
            const long long nx = by_mask ? r.nm : r.nc, ny = by_mask ? r.nc : r.nm;
            const V* v = val + rp[i];
            const long long out = rpo[i];
            IT j[4];
            long long at[4];
            bool stays[4];
            filter_entries<WARPS>(
                nx, w,
                [&](long long q, int stride) {
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        j[u] = q + u * stride < nx ? x[q + u * stride] : IT(-1);
                    lower_bound4<IT>(y, ny, j, at);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        stays[u] = (at[u] < ny && y[at[u]] == j[u]) != (complement != 0);
                        if (!by_mask) at[u] = q + u * stride;   // the entry's place in C(i,:)
                    }
                },
                [&](int u) { return stays[u]; },
                [&](int u, long long pos) {
                    colo[out + pos] = j[u];
                    if constexpr (HV) valo[out + pos] = v[at[u]];
                });
        });
}

}  // namespace sg

namespace {

spgemm_status kfail(spgemm_status st, const char* msg) {
    sg::set_last_error(msg);
    return st;
}

spgemm_status kcheck(const spgemm_csr* C, const spgemm_csr* M) {
    if (!C || !M || !C->rowptr || !M->rowptr || C->nrows < 0 ||
        (C->nnz > 0 && !C->col) || (M->nnz > 0 && !M->col))
        return kfail(SPGEMM_ERR_INVALID_ARG, "mask: NULL or malformed matrix");
    if (M->nrows != C->nrows || M->ncols != C->ncols)
        return kfail(SPGEMM_ERR_INVALID_ARG, "mask: M and C differ in shape");
    if (M->index_type != C->index_type)
        return kfail(SPGEMM_ERR_INVALID_ARG, "mask: M and C differ in index type");
    if (C->value_type != SPGEMM_BOOL && C->nnz > 0 && !C->val)
        return kfail(SPGEMM_ERR_INVALID_ARG, "mask: C has no values");
    return SPGEMM_OK;
}

unsigned grid_rows(long long m) {
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return (unsigned)std::max<long long>(1, std::min<long long>((m + 7) / 8, (long long)sms * 8));
}

}  // namespace

extern "C" {

size_t spgemm_mask_workspace_size(int64_t m) {
    if (m < 0) m = 0;
    return sg::scan_temp_bytes(m + 1);
}

spgemm_status spgemm_mask_count(const spgemm_csr* C, const spgemm_csr* M, int32_t complement,
                                void* stream, void* ws, size_t ws_bytes, int64_t* rowptrP,
                                int64_t* nnz_host) {
    sg::set_last_error("");
    spgemm_status st = kcheck(C, M);
    if (st != SPGEMM_OK) return st;
    const long long m = C->nrows;
    if (!rowptrP || !nnz_host || !ws || ws_bytes < spgemm_mask_workspace_size(m))
        return kfail(SPGEMM_ERR_INVALID_ARG, "mask: outputs or workspace missing");
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaMemsetAsync(rowptrP + m, 0, 8, s);
    if (e == cudaSuccess && m > 0) {
        sg::count_launches(1);
        if (C->index_type == SPGEMM_INDEX_I32)
            sg::mask_count_kernel<int32_t><<<grid_rows(m), 256, 0, s>>>(
                m, C->rowptr, C->rowend, (const int32_t*)C->col, M->rowptr, M->rowend,
                (const int32_t*)M->col, complement, rowptrP);
        else
            sg::mask_count_kernel<int64_t><<<grid_rows(m), 256, 0, s>>>(
                m, C->rowptr, C->rowend, (const int64_t*)C->col, M->rowptr, M->rowend,
                (const int64_t*)M->col, complement, rowptrP);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = sg::launch_exclusive_scan(rowptrP, m + 1, (int64_t*)ws, s);
    int64_t total = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&total, rowptrP + m, 8, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return kfail(SPGEMM_ERR_CUDA, cudaGetErrorString(e));
    *nnz_host = total;
    return SPGEMM_OK;
}

spgemm_status spgemm_mask_fill(const spgemm_csr* C, const spgemm_csr* M, int32_t complement,
                               void* stream, const int64_t* rowptrP, void* colP, void* valP) {
    sg::set_last_error("");
    spgemm_status st = kcheck(C, M);
    if (st != SPGEMM_OK) return st;
    const long long m = C->nrows;
    if (!rowptrP) return kfail(SPGEMM_ERR_INVALID_ARG, "mask: rowptrP is NULL");
    if (m == 0) return SPGEMM_OK;
    cudaStream_t s = (cudaStream_t)stream;
    const int vt = C->value_type;
    const bool i32 = C->index_type == SPGEMM_INDEX_I32;
    cudaError_t e = sg::with_value_type(vt, [&](auto tag) -> cudaError_t {
        using V = decltype(tag);
        sg::count_launches(1);
        if (i32)
            sg::mask_fill_kernel<int32_t, V><<<grid_rows(m), 256, 0, s>>>(
                m, C->rowptr, C->rowend, (const int32_t*)C->col, (const V*)C->val, M->rowptr,
                M->rowend, (const int32_t*)M->col, complement, rowptrP, (int32_t*)colP, (V*)valP);
        else
            sg::mask_fill_kernel<int64_t, V><<<grid_rows(m), 256, 0, s>>>(
                m, C->rowptr, C->rowend, (const int64_t*)C->col, (const V*)C->val, M->rowptr,
                M->rowend, (const int64_t*)M->col, complement, rowptrP, (int64_t*)colP, (V*)valP);
        return cudaGetLastError();
    });
    if (e != cudaSuccess) return kfail(SPGEMM_ERR_CUDA, cudaGetErrorString(e));
    return SPGEMM_OK;
}

}  // extern "C"
