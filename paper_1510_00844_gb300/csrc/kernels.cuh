// Kernels of the two-phase sparse product C = A.B (Gustavson, Alg. 1, on
// CSR rows) and the k-slice bounds (Sec. 4.1).  Templates over the column
// index type IT (int32_t / int64_t) and the value type V (double, float,
// int64_t, the min-semiring wrappers, NoVal for the Boolean semiring).
//
// Row classes (decided from flops_i = sum_{k in A(i,:)} nnz(B(k,:)), Sec. 2):
//   EMPTY       flops_i == 0
//   HASH(b)     flops_i <= dense_min (<= 1024).  Up to 32 products: one warp
//               per row in registers (equal columns by match).  33 to 128 and n
//               < 2^25, numeric: one warp per row, products sorted in
//               registers by (column, position); likewise 129 to 512 and n <
//               2^23 outside the persistent chain and predicted slots.  Other
//               rows of 129 to 1024 and n within rank_max_n, outside the
//               chain: one block per row, columns ranked by a bitmap of n bits
//               in shared memory.
//               Otherwise: one warp per row with a warp-private hash table in
//               shared memory, output sorted in the warp (bitonic sort up to
//               64 entries, stable radix sort above).
//   DENSE(b)    flops_i > dense_min: symbolic = one block per row with a
//               bitmap of all n columns in shared memory (also yields
//               per-chunk counts; kept in the workspace for patterns, whose
//               numeric phase writes the columns from it); numeric = one warp
//               per (row, column segment) sweeping column chunks with a dense
//               accumulator, so the output comes out sorted.  DENSE rows are
//               bucketed by floor(log2 flops_i), largest first.
#pragma once

#include "device_common.cuh"
#include "rows.cuh"

namespace sg {

constexpr int kNumHashBins = 4;
__host__ __device__ constexpr int hash_bin_flops(int b) {
    return b == 0 ? 32 : b == 1 ? 128 : b == 2 ? 512 : 1024;
}
constexpr int kDenseMinLog2 = 10;  // flops > 1024 -> dense
constexpr int kDenseMaxLog2 = 40;
constexpr int kClassEmpty = 0;
constexpr int kClassHash0 = 1;
constexpr int kClassDense0 = kClassHash0 + kNumHashBins;          // largest-flops bucket
constexpr int kNumClasses = kClassDense0 + (kDenseMaxLog2 - kDenseMinLog2 + 1);
constexpr int kSegGrid = 16;
// Table size (log2 slots) of hash bin 0, whose rows (at most 32 products)
// take the table-free short-row path instead.
constexpr int kShortLog2T = 6;
// Dense chunk configurations (columns per chunk, warps per block): one is
// chosen per plan (spgemm_opts.dense_chunk forces one).
constexpr int kDenseW0 = 1024, kDenseWarps0 = 8;
constexpr int kDenseW1 = 2048, kDenseWarps1 = 4;

// One product of a batch (C_p = A_p . B_p).  Rows of all products are
// numbered globally: product p owns global rows [row_base, row_base + m) and
// global B rows [brow_base, brow_base + l).  The workspace offsets give each
// product its slice of the shared tables.
struct ProdDesc {
    long long m, l, n;
    long long row_base, brow_base;
    const int64_t* rpA;
    const int64_t* reA;
    const void* ciA;
    const void* vA;
    const int64_t* rpB;
    const void* ciB;
    const void* vB;
    long long nnzB;
    long long chunk_base;  // dense chunk counts: chunk_base + i * P + c
    long long seg_base;    // segment table: seg_base + k * (kSegGrid + 1) + g
    long long run_base;    // run lengths: run_base + q (q a position in B's arrays)
    int P;                 // column chunks per row
    int pad;
};

constexpr int kMaxDenseClasses = kDenseMaxLog2 - kDenseMinLog2 + 1;

struct DevCounters {
    unsigned long long class_count[kNumClasses];
    unsigned long long class_cursor[kNumClasses];
    unsigned long long class_off[kNumClasses + 1];
    unsigned long long unit_begin[kMaxDenseClasses + 1];  // dense work units per class
    unsigned long long total_flops;
    unsigned long long max_flops;
    unsigned long long work_counter[4];  // dynamic row grabbing
    unsigned long long max_dense_len;    // longest A row among dense rows
    int64_t nnz_c;                       // total of the row pointers, read back with err
    int err;
    int unsupported;
    int seg_log2;                        // dense work-unit size of the plan
    unsigned blocks_done;                // of the row analysis
    int pad[26];
};

// Product owning global row r: the largest p with rb[p] <= r.
__device__ __forceinline__ int find_prod(const long long* __restrict__ rb, int nprod, long long r) {
    int lo = 0, hi = nprod - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (rb[mid] <= r) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Everything a kernel needs about global row r.
template <class IT, class V>
struct RowCtx {
    long long i, a0, a1, n;
    const IT* ciA;
    const V* vA;
    const int64_t* rpB;
    const IT* ciB;
    const V* vB;
    long long chunk_base, seg_base, run_base;
    int P;
};

template <class IT, class V>
__device__ __forceinline__ RowCtx<IT, V> row_ctx(const ProdDesc* __restrict__ D,
                                                 const long long* __restrict__ rb, int nprod,
                                                 long long r) {
    const int p = nprod > 1 ? find_prod(rb, nprod, r) : 0;
    const ProdDesc& d = D[p];
    RowCtx<IT, V> c;
    c.i = r - d.row_base;
    c.a0 = d.rpA[c.i];
    c.a1 = d.reA ? d.reA[c.i] : d.rpA[c.i + 1];
    c.n = d.n;
    c.ciA = (const IT*)d.ciA;
    c.vA = (const V*)d.vA;
    c.rpB = d.rpB;
    c.ciB = (const IT*)d.ciB;
    c.vB = (const V*)d.vB;
    c.chunk_base = d.chunk_base;
    c.seg_base = d.seg_base;
    c.run_base = d.run_base;
    c.P = d.P;
    return c;
}

// The rows rows[first], rows[first + stride], ... (< nrows) of a class,
// walked by one warp.  (Loading the next rows' ids and bounds while a row is
// processed was measured on the short rows of the AMG hierarchy and gained
// nothing.)
template <class IT, class V, class F>
__device__ __forceinline__ void for_class_rows(const ProdDesc* __restrict__ D,
                                               const long long* __restrict__ rb, int nprod,
                                               const int32_t* __restrict__ crow, long long first,
                                               long long nrows, long long stride, F&& f) {
    for (long long rr = first; rr < nrows; rr += stride) {
        const long long r = crow[rr];
        f(row_ctx<IT, V>(D, rb, nprod, r), r);
    }
}

// Rows [r0, r1) of a block by class: with base == nullptr, count them per
// class into loc; else place row r at base[c] + a slot taken from loc[c].
// Lanes of a warp with the same class take one atomic together.
__device__ __forceinline__ void bin_block_rows(const unsigned char* __restrict__ cls,
                                               int32_t* __restrict__ rows, long long r0,
                                               long long r1, unsigned long long* loc,
                                               const unsigned long long* base) {
    const int lane = threadIdx.x & 31;
    for (long long b = r0 + (threadIdx.x & ~31); b < r1; b += blockDim.x) {
        const long long r = b + lane;
        const bool valid = r < r1;
        const int c = valid ? (int)cls[r] : -1 - lane;
        const unsigned grp = __match_any_sync(0xffffffffu, c);
        const int leader = __ffs(grp) - 1;
        const int rank = __popc(grp & ((1u << lane) - 1u));
        unsigned long long first = 0;
        if (valid && lane == leader) first = atomicAdd(&loc[c], (unsigned long long)__popc(grp));
        first = __shfl_sync(0xffffffffu, first, leader);
        if (valid && base) rows[base[c] + first + rank] = (int32_t)r;
    }
}

// Tile of the int64 exclusive scan: 256 threads x 16 items.
constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int kScanTile = kScanThreads * kScanItems;

// Class of a row with `flops` products: EMPTY, the smallest hash bin that
// holds flops << hash_shift while flops <= dense_min (<= 1024; the largest
// bin takes the rest), else the dense bucket of floor(log2 flops), largest
// first.
__host__ __device__ __forceinline__ int row_class(long long flops, int dense_min,
                                                  int hash_shift = 0) {
    if (flops == 0) return kClassEmpty;
    if (flops <= dense_min) {
#pragma unroll
        for (int b = 0; b < kNumHashBins - 1; ++b)
            if ((flops << hash_shift) <= hash_bin_flops(b)) return kClassHash0 + b;
        return kClassHash0 + kNumHashBins - 1;
    }
#ifdef __CUDA_ARCH__
    int lg = 63 - __clzll(flops);
#else
    int lg = 63 - __builtin_clzll((unsigned long long)flops);
#endif
    if (lg > kDenseMaxLog2) lg = kDenseMaxLog2;
    if (lg < kDenseMinLog2) lg = kDenseMinLog2;
    return kClassDense0 + (kDenseMaxLog2 - lg);
}

// Segments per row of dense class t (floor(log2 flops) = kDenseMaxLog2 - t):
// about 2^seg_log2 products per segment (a plan knob; by default chosen from
// the plan's flops so that big products get fewer, longer units), at most
// kSegGrid.
__host__ __device__ __forceinline__ int dense_class_segments(int t, int seg_log2) {
    const int lg = kDenseMaxLog2 - t;
    int sh = lg + 1 - seg_log2;
    if (sh < 0) sh = 0;
    if (sh > 4) sh = 4;  // kSegGrid = 16
    return 1 << sh;
}

// Class offsets (exclusive scan of the counts) and the dense work-unit prefix,
// by one warp.
__device__ __forceinline__ void class_offsets(DevCounters* cnt, int seg_log2) {
    const int lane = lane_id();
    if (lane == 0) cnt->seg_log2 = seg_log2;
    static_assert(kNumClasses <= 64 && kMaxDenseClasses < 32, "two classes, one dense class per lane");
    unsigned long long base = 0;
    for (int c0 = 0; c0 < kNumClasses; c0 += 32) {
        const int c = c0 + lane;
        const unsigned long long n = c < kNumClasses ? __ldcg(&cnt->class_count[c]) : 0ull;
        const unsigned long long incl = warp_incl_scan(n);
        if (c < kNumClasses) {
            cnt->class_cursor[c] = base + incl - n;
            cnt->class_off[c] = base + incl - n;
        }
        base += __shfl_sync(kFull, incl, 31);
    }
    if (lane == 0) cnt->class_off[kNumClasses] = base;
    const unsigned long long u =
        lane < kMaxDenseClasses
            ? __ldcg(&cnt->class_count[kClassDense0 + lane]) * dense_class_segments(lane, seg_log2)
            : 0ull;
    const unsigned long long incl = warp_incl_scan(u);
    if (lane <= kMaxDenseClasses) cnt->unit_begin[lane] = incl - u;
}

__device__ __forceinline__ long long row_end(const int64_t* rp, const int64_t* re, long long i) {
    return re ? re[i] : rp[i + 1];
}

// ----------------------------------------------------------------- K1: flops
// Per global row (a warp per tile of 32 rows): flops_i, its class, per-class
// counts, total and max flops, longest dense row; a product whose dense rows
// need more columns than the shared-memory bitmap holds is flagged.
// What bounds it: the longest rows, walked by one warp with eight entries per
// lane in flight (with one, the 240 us of an R-MAT 18 analysis were its longest
// row's 250 dependent steps; now 150 us).
// Learned sizing (not in the paper): when `prm` is given, the row-size predictor
// is evaluated on each row's features (a lane per row: with a lane per
// hidden unit, row after row, 40009 rows took 286 us; now 25 us), which gives
// the predicted capacity cap_out[r] = clamp(2^(y +
// margin) - 1, max_k |B(k,:)|, min(flops, n)), and bins rows of at most
// dense_min products by that capacity instead of by their flops.
constexpr int kSizerF = 6;

// The row-size predictor on one row's features, by one lane; prm: W1 (32 x F),
// b1, W2 (32 x 32), b2, w3, b3.  Products are rounded and added in ascending
// input; the last layer's 32 terms are added as a tree over i, i + 16; i, i + 8;
// ... so that a warp that holds one unit per lane gets the same sum.
__device__ __forceinline__ float sizer_eval(const float* prm, const float (&x)[kSizerF]) {
    const float* W1 = prm;
    const float* b1 = W1 + 32 * kSizerF;
    const float* W2 = b1 + 32;
    const float* b2 = W2 + 32 * 32;
    const float* w3 = b2 + 32;
    float h1[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        float z = b1[j];
#pragma unroll
        for (int q = 0; q < kSizerF; ++q) z = __fadd_rn(z, __fmul_rn(W1[j * kSizerF + q], x[q]));
        h1[j] = z > 0.f ? z : 0.f;
    }
    // the terms of units j and j + 16 together, so that the tree's first level
    // needs no array of 32 terms
    float term[16];
#pragma unroll 4
    for (int j = 0; j < 16; ++j) {
        float z = b2[j], y = b2[j + 16];
#pragma unroll
        for (int k = 0; k < 32; ++k) {
            z = __fadd_rn(z, __fmul_rn(W2[j * 32 + k], h1[k]));
            y = __fadd_rn(y, __fmul_rn(W2[(j + 16) * 32 + k], h1[k]));
        }
        term[j] = __fadd_rn(__fmul_rn(w3[j], z > 0.f ? z : 0.f),
                            __fmul_rn(w3[j + 16], y > 0.f ? y : 0.f));
    }
#pragma unroll
    for (int d = 8; d; d >>= 1)
#pragma unroll
        for (int j = 0; j < d; ++j) term[j] = __fadd_rn(term[j], term[j + d]);
    return term[0] + w3[32];
}

template <class IT, bool PREDICT>
__device__ __forceinline__ void analyze_kernel_body(long long R, const ProdDesc* __restrict__ D,
                               const long long* __restrict__ rb, int nprod, long long max_dense_n,
                               int dense_min, int64_t* __restrict__ flops_out,
                               unsigned char* __restrict__ cls_out, DevCounters* cnt,
                               const float* __restrict__ prm, float margin,
                               int64_t* __restrict__ cap_out, int hash_shift, int tile_rows,
        const long long vbid, const long long vnb) {
    __shared__ unsigned long long hist[kNumClasses];
    __shared__ unsigned long long blk_total, blk_max, blk_dlen;
    __shared__ int blk_unsup;
    constexpr int kParams = 32 * kSizerF + 32 + 32 * 32 + 32 + 32 + 1;
    __shared__ float sp[PREDICT ? kParams : 1];
    if constexpr (PREDICT)
        for (int q = threadIdx.x; q < kParams; q += blockDim.x) sp[q] = prm[q];
    for (int t = threadIdx.x; t < kNumClasses; t += blockDim.x) hist[t] = 0;
    if (threadIdx.x == 0) {
        blk_total = 0;
        blk_max = 0;
        blk_dlen = 0;
        blk_unsup = 0;
    }
    __syncthreads();
    const int lane = lane_id();
    const long long warp = ((long long)vbid * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)vnb * blockDim.x) >> 5;
    unsigned long long my_total = 0, my_max = 0;
    // Tiles of tile_rows <= 32 rows (fewer where there are few rows for the
    // warps): a row of at most 32 A entries is summed by its own lane (eight
    // entries' loads in flight at a time); longer rows by the whole warp, one
    // after another.
    for (long long tile = warp; tile * tile_rows < R; tile += nwarps) {
        const long long r = tile * tile_rows + lane;
        const bool in = lane < tile_rows && r < R;
        RowCtx<IT, NoVal> c{};
        if (in) c = row_ctx<IT, NoVal>(D, rb, nprod, r);
        const long long d = in ? c.a1 - c.a0 : 0;
        long long f = 0, mx = 0;
        if (in && d <= 32) {
            for (long long p0 = c.a0; p0 < c.a1; p0 += 8) {
                long long k[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) k[u] = p0 + u < c.a1 ? (long long)c.ciA[p0 + u] : -1;
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    if (k[u] >= 0) {
                        const long long len = c.rpB[k[u] + 1] - c.rpB[k[u]];
                        f += len;
                        mx = len > mx ? len : mx;
                    }
                }
            }
        }
        for (unsigned lm = __ballot_sync(kFull, in && d > 32); lm; lm &= lm - 1u) {
            const int src = __ffs(lm) - 1;
            const RowCtx<IT, NoVal> cs = row_ctx<IT, NoVal>(D, rb, nprod, tile * tile_rows + src);
            long long fs = 0, ms = 0;
            for (long long p = cs.a0 + lane; p < cs.a1; p += 256) {
                long long k[8];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    k[u] = p + 32 * u < cs.a1 ? (long long)cs.ciA[p + 32 * u] : -1;
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (k[u] >= 0) {
                        const long long len = cs.rpB[k[u] + 1] - cs.rpB[k[u]];
                        fs += len;
                        ms = len > ms ? len : ms;
                    }
            }
            fs = warp_sum(fs);
            ms = warp_max(ms);
            if (lane == src) {
                f = fs;
                mx = ms;
            }
        }
        long long cap = 0;
        if (PREDICT && in && f > 0) {
            const long long ub = f < c.n ? f : c.n;
            const float x[kSizerF] = {log2f(1.f + (float)f),    log2f(1.f + (float)d),
                                      log2f(1.f + (float)mx),   log2f(1.f + (float)c.n),
                                      log2f(1.f + (float)f / (float)d), log2f(1.f + (float)ub)};
            const float est = exp2f(sizer_eval(sp, x) + margin) - 1.f;
            cap = est >= (float)ub ? ub : (long long)ceilf(est > 0.f ? est : 0.f);
            if (cap < mx) cap = mx;
            if (cap > ub) cap = ub;
        }
        int cl = -1 - lane;
        if (in) {
            flops_out[r] = f;
            if (cap_out) cap_out[r] = PREDICT ? cap : f;
            cl = row_class(f, dense_min, hash_shift);
            if (PREDICT && cl > kClassEmpty && cl < kClassDense0) {
                cl = row_class(cap > 0 ? cap : 1, dense_min, hash_shift);
                // bin 0 is the short-row path (one product per lane): a row
                // with more products takes bin 1's table whatever its size
                if (cl == kClassHash0 && f > 32) cl = kClassHash0 + 1;
            }
            cls_out[r] = (unsigned char)cl;
            if (cl >= kClassDense0) {
                if (c.n > max_dense_n) blk_unsup = 1;
                atomicMax(&blk_dlen, (unsigned long long)d);
            }
            my_total += (unsigned long long)f;
            if ((unsigned long long)f > my_max) my_max = (unsigned long long)f;
        }
        // one shared atomic per class present in the tile
        const unsigned grp = __match_any_sync(kFull, cl);
        if (in && (grp & lanemask_lt()) == 0u) atomicAdd(&hist[cl], (unsigned long long)__popc(grp));
    }
    my_total = warp_sum(my_total);
    my_max = warp_max(my_max);
    if (lane == 0) {
        atomicAdd(&blk_total, my_total);
        atomicMax(&blk_max, my_max);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < kNumClasses; t += blockDim.x)
        if (hist[t]) atomicAdd(&cnt->class_count[t], hist[t]);
    if (threadIdx.x == 0) {
        atomicAdd(&cnt->total_flops, blk_total);
        atomicMax(&cnt->max_flops, blk_max);
        atomicMax(&cnt->max_dense_len, blk_dlen);
        if (blk_unsup) atomicExch(&cnt->unsupported, 1);
    }
}

// The last block to finish also forms the class offsets.
template <class IT, bool PREDICT>
__global__ void __launch_bounds__(256) analyze_kernel(long long R, const ProdDesc* __restrict__ D,
                               const long long* __restrict__ rb, int nprod, long long max_dense_n,
                               int dense_min, int64_t* __restrict__ flops_out,
                               unsigned char* __restrict__ cls_out, DevCounters* cnt,
                               const float* __restrict__ prm, float margin,
                               int64_t* __restrict__ cap_out, int hash_shift, int tile_rows,
                               int seg_log2) {
    analyze_kernel_body<IT, PREDICT>(R, D, rb, nprod, max_dense_n, dense_min, flops_out, cls_out, cnt,
        prm, margin, cap_out, hash_shift, tile_rows, (long long)blockIdx.x, (long long)gridDim.x);
    __shared__ bool last;
    __threadfence();   // this thread's counts come before the block's ticket
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&cnt->blocks_done, 1u) + 1u == gridDim.x;
    __syncthreads();
    if (last && threadIdx.x < 32) class_offsets(cnt, seg_log2);
}

// Features of every global row for the row-size predictor (log2(1 + .) of
// flops, |A(i,:)|, max_k |B(k,:)|, n, flops/|A(i,:)|, min(flops, n)).
template <class IT>
__global__ void row_features_kernel(long long R, const ProdDesc* __restrict__ D,
                                    const long long* __restrict__ rb, int nprod,
                                    float* __restrict__ X) {
    const int lane = lane_id();
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long r = warp; r < R; r += nwarps) {
        const RowCtx<IT, NoVal> c = row_ctx<IT, NoVal>(D, rb, nprod, r);
        long long f = 0, mx = 0;
        for (long long p = c.a0 + lane; p < c.a1; p += 32) {
            long long k = (long long)c.ciA[p];
            const long long len = c.rpB[k + 1] - c.rpB[k];
            f += len;
            mx = len > mx ? len : mx;
        }
        f = warp_sum(f);
        mx = warp_max(mx);
        if (lane == 0) {
            const long long d = c.a1 - c.a0;
            const long long ub = f < c.n ? f : c.n;
            float* x = X + r * kSizerF;
            x[0] = log2f(1.f + (float)f);
            x[1] = log2f(1.f + (float)d);
            x[2] = log2f(1.f + (float)mx);
            x[3] = log2f(1.f + (float)c.n);
            x[4] = log2f(1.f + (d > 0 ? (float)f / (float)d : 0.f));
            x[5] = log2f(1.f + (float)ub);
        }
    }
}

// ----------------------------------------------------------- checked mode
// One warp per row: rowptr monotone, columns in [0, ncols), strictly ascending.
template <class IT>
__global__ void validate_kernel(long long m, long long ncols, long long nnz, const int64_t* rp,
                                const int64_t* re, const IT* ci, int* err) {
    const int lane = lane_id();
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long i = warp; i < m; i += nwarps) {
        long long a0 = rp[i], a1 = row_end(rp, re, i);
        if (a0 < 0 || a1 < a0 || a1 > nnz || (!re && i == 0 && a0 != 0)) {
            if (lane == 0) atomicExch(err, (int)kDevBadRowptr);
            continue;
        }
        for (long long p = a0 + lane; p < a1; p += 32) {
            long long c = (long long)ci[p];
            bool bad = c < 0 || c >= ncols || (p + 1 < a1 && (long long)ci[p + 1] <= c);
            if (bad) atomicExch(err, (int)kDevBadIndex);
        }
    }
}

// ------------------------------------------ short rows (hash bin 0)
// A row of at most 32 products needs no table.  Lane x takes the row's x-th
// product in ascending k (then in B(k,:)'s order): the A entries are read in
// batches of 32 and each batch's products are flattened onto the lanes after
// those of earlier batches; the owner of product f is the last entry whose
// exclusive prefix of run lengths is <= f (a five-step search over the
// lanes, always a lane of the batch).  Equal columns are then grouped with
// __match_any_sync.  Returns the number of products, or -1 if the row has
// more than 32 (a row of hash bin 0 never does).
template <class IT, class V, bool VALS>
__device__ __forceinline__ int short_row_gather(const RowCtx<IT, V>& c,
                                                typename KeyT<IT>::type& key, V& v) {
    using K = typename KeyT<IT>::type;
    const int lane = lane_id();
    int have = 0;
    key = K(-1);
    v = VOps<V>::init();
    for (long long b = c.a0; b < c.a1; b += 32) {
        const int nb = (int)min(32LL, c.a1 - b);
        long long lo = 0;
        int len = 0;
        V a = VOps<V>::init();
        if (lane < nb) {
            const long long k = (long long)c.ciA[b + lane];
            lo = c.rpB[k];
            // capped: more than 32 products in one B row already makes the
            // row too long for this path, and keeps the scan in int range
            len = (int)min(c.rpB[k + 1] - lo, 33LL);
            if constexpr (VALS) a = load_val(c.vA, b + lane);
        }
        const int incl = warp_incl_scan(len);
        const int tot = __shfl_sync(kFull, incl, 31);
        if (tot == 0) continue;
        if (have + tot > 32) return -1;
        const int excl = incl - len;
        const int f = lane - have;
        int e = 0;
#pragma unroll
        for (int w = 16; w; w >>= 1) {
            const int cand = e + w;
            const int ex = __shfl_sync(kFull, excl, cand & 31);
            if (cand < nb && ex <= f) e = cand;
        }
        const long long lo_e = __shfl_sync(kFull, lo, e);
        const int ex_e = __shfl_sync(kFull, excl, e);
        const V a_e = shfl_val(a, e);
        if (f >= 0 && f < tot) {
            const long long q = lo_e + (f - ex_e);
            key = (K)c.ciB[q];
            if constexpr (VALS) v = VOps<V>::mul(a_e, load_val(c.vB, q));
        }
        have += tot;
    }
    return have;
}

// Symbolic count of a short row: the number of distinct columns.
template <class IT>
__device__ __forceinline__ void short_row_symbolic(const RowCtx<IT, NoVal>& c, long long r,
                                                   int64_t* __restrict__ rowcnt, int* err) {
    using K = typename KeyT<IT>::type;
    const int lane = lane_id();
    K key;
    NoVal v;
    const int np = short_row_gather<IT, NoVal, false>(c, key, v);
    if (np < 0) {
        if (lane == 0) atomicExch(err, (int)kDevTableFull);
        return;
    }
    const bool valid = lane < np;
    const K kk = valid ? key : (K)(-1 - lane);
    const unsigned grp = __match_any_sync(kFull, kk);
    const bool leader = valid && (grp & lanemask_lt()) == 0u;
    const int cnt = __popc(__ballot_sync(kFull, leader));
    if (lane == 0) rowcnt[r] = cnt;
}

// Numeric pass of a short row: the lowest lane of each group of equal
// columns adds the group's products in lane order from the identity (the
// order in which the hash path adds them), and writes its column at the
// number of groups with a smaller column.  Slot mode as in the hash path.
template <class IT, class V>
__device__ __forceinline__ void short_row_numeric(const RowCtx<IT, V>& c, long long r,
                                                  const int64_t* __restrict__ rpC, long long cap,
                                                  IT* __restrict__ ciC, V* __restrict__ vC,
                                                  int* err, int64_t* __restrict__ rowend,
                                                  int32_t* __restrict__ overflow,
                                                  unsigned* overflow_count) {
    using K = typename KeyT<IT>::type;
    constexpr bool HV = VOps<V>::has_val;
    const int lane = lane_id();
    // the output range does not depend on the products: loaded first
    const long long out = rpC[r];
    long long rcnt = rpC[r + 1] - out;
    K key;
    V v;
    const int np = short_row_gather<IT, V, HV>(c, key, v);
    if (np < 0) {
        if (lane == 0) atomicExch(err, (int)kDevTableFull);
        return;
    }
    const bool valid = lane < np;
    const K kk = valid ? key : (K)(-1 - lane);
    const unsigned grp = __match_any_sync(kFull, kk);
    const bool leader = valid && (grp & lanemask_lt()) == 0u;
    const unsigned L = __ballot_sync(kFull, leader);
    const int cnt = __popc(L);
    V sum = VOps<V>::init();
    if constexpr (HV) {
        unsigned rem = leader ? grp : 0u;
        const int maxc = (int)__reduce_max_sync(kFull, (unsigned)__popc(rem));
        for (int t = 0; t < maxc; ++t) {
            const int src = rem ? __ffs(rem) - 1 : lane;
            const V x = shfl_val(v, src);
            if (rem) {
                sum = VOps<V>::add(sum, x);
                rem &= rem - 1u;
            }
        }
    }
    int pos = 0;
    for (unsigned Lr = L; Lr; Lr &= Lr - 1u) {
        const K kj = __shfl_sync(kFull, kk, __ffs(Lr) - 1);
        pos += kj < kk ? 1 : 0;
    }
    if (rowend != nullptr) {
        if (cnt > rcnt) {
            if (lane == 0) {
                overflow[atomicAdd(overflow_count, 1u)] = (int32_t)r;
                rowend[r] = -1;
            }
            return;
        }
        rcnt = cnt;
        if (lane == 0) rowend[r] = out + cnt;
    } else if (cnt != rcnt && lane == 0) {
        atomicExch(err, (int)kDevCountMismatch);
    }
    if (out + rcnt > cap && lane == 0) atomicExch(err, (int)kDevCapacity);
    if (leader && pos < rcnt && out + pos < cap) {
        ciC[out + pos] = (IT)kk;
        if constexpr (HV) vC[out + pos] = sum;
    }
}

// ------------------------------ rows of at most 128 products, sorted
// The products of a row of at most 32 * ITEMS products are spread over the
// lanes in ascending k (product f to lane f % 32, item f / 32), sorted by
// (column, f) in registers -- a bitonic network on 32-bit keys that hold both,
// so columns must be below 2^(32 - bits of f) -- and each run of equal columns
// is added up by its first lane, in ascending f.  Nothing depends on a table:
// no probes, no compaction, no slots to clear, and a 32-bit exchange instead of
// a sort of (column, value) pairs in shared memory.  Rows of 56 products (R^T A
// of a 128^3 grid): 1459 warp instructions per row with the table, 670 with
// this; the pass over 262144 of them 0.55 -> 0.33 ms.  (Rows of at most 32 products
// are no faster this way: they wait for their scattered loads.)
template <int ITEMS>
constexpr int kSortBits = ITEMS == 2 ? 6 : 7;

// Whether a product of n columns can be sorted this way (the largest key is
// kept for places without a product).
template <int ITEMS>
__device__ __forceinline__ bool sortable_columns(long long n) {
    return n < (1LL << (32 - kSortBits<ITEMS>));
}

// Gathers the row's products: their (column, f) keys to registers, their
// values to vals[f].  Returns how many there are, or -1 if more than
// 32 * ITEMS (vals then holds some of them).
template <class IT, class V, int ITEMS>
__device__ __forceinline__ int sorted_row_gather(const RowCtx<IT, V>& c, unsigned (&key)[ITEMS],
                                                 V* vals) {
    constexpr bool HV = VOps<V>::has_val;
    constexpr int B = kSortBits<ITEMS>;
    const int lane = lane_id();
    int have = 0;
#pragma unroll
    for (int t = 0; t < ITEMS; ++t) key[t] = 0xffffffffu;
    for (long long b = c.a0; b < c.a1; b += 32) {
        const int nb = (int)min(32LL, c.a1 - b);
        long long lo = 0;
        int len = 0;
        V a = VOps<V>::init();
        if (lane < nb) {
            const long long k = (long long)c.ciA[b + lane];
            lo = c.rpB[k];
            // capped: one such B row already makes the row too long, and the
            // scan stays in int range
            len = (int)min(c.rpB[k + 1] - lo, 32LL * ITEMS + 1);
            if constexpr (HV) a = load_val(c.vA, b + lane);
        }
        const int incl = warp_incl_scan(len);
        const int tot = __shfl_sync(kFull, incl, 31);
        if (tot == 0) continue;
        if (have + tot > 32 * ITEMS) return -1;
        const int excl = incl - len;
#pragma unroll
        for (int t = 0; t < ITEMS; ++t) {
            if (32 * t + 31 < have || 32 * t >= have + tot) continue;
            const int f = 32 * t + lane - have;
            // the owner of f: the last entry whose exclusive prefix is <= f
            int e = 0;
#pragma unroll
            for (int w = 16; w; w >>= 1) {
                const int cand = e + w;
                const int ex = __shfl_sync(kFull, excl, cand & 31);
                if (cand < nb && ex <= f) e = cand;
            }
            const long long q = __shfl_sync(kFull, lo, e) + (f - __shfl_sync(kFull, excl, e));
            const V a_e = shfl_val(a, e);
            if (f >= 0 && f < tot) {
                key[t] = (unsigned)c.ciB[q] << B | (unsigned)(32 * t + lane);
                if constexpr (HV) vals[32 * t + lane] = VOps<V>::mul(a_e, load_val(c.vB, q));
            }
        }
        have += tot;
    }
    return have;
}

// Ascending bitonic sort of the warp's 32 * ITEMS keys (key 32 * t + lane in
// item t of a lane).
template <int ITEMS>
__device__ __forceinline__ void warp_sort_keys(unsigned (&key)[ITEMS]) {
    const int lane = lane_id();
#pragma unroll
    for (int k = 2; k <= 32 * ITEMS; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j >= 32) {
#pragma unroll
                for (int t = 0; t < ITEMS; ++t) {
                    const int o = t ^ (j >> 5);
                    if (o > t) {
                        const unsigned x = min(key[t], key[o]), y = max(key[t], key[o]);
                        const bool up = (32 * t & k) == 0;
                        key[t] = up ? x : y;
                        key[o] = up ? y : x;
                    }
                }
            } else {
#pragma unroll
                for (int t = 0; t < ITEMS; ++t) {
                    const unsigned y = __shfl_xor_sync(kFull, key[t], j);
                    const bool up = ((32 * t + lane) & k) == 0;
                    const bool lower = (lane & j) == 0;
                    key[t] = up == lower ? min(key[t], y) : max(key[t], y);
                }
            }
        }
    }
}

// Numeric pass of such a row (np products, gathered): sorted, reduced, written.
// `sorted` is room for 32 * ITEMS keys.  Slot mode as in the hash path.
template <class IT, class V, int ITEMS>
__device__ __forceinline__ void sorted_row_numeric(unsigned (&key)[ITEMS], int np, long long r,
                                                   const V* vals, unsigned* sorted,
                                                   const int64_t* __restrict__ rpC, long long cap,
                                                   IT* __restrict__ ciC, V* __restrict__ vC,
                                                   int* err, int64_t* __restrict__ rowend,
                                                   int32_t* __restrict__ overflow,
                                                   unsigned* overflow_count) {
    constexpr bool HV = VOps<V>::has_val;
    constexpr int B = kSortBits<ITEMS>;
    constexpr unsigned kPlace = 32 * ITEMS - 1;
    constexpr bool kPlain = std::is_same<V, double>::value || std::is_same<V, float>::value ||
                            std::is_same<V, int64_t>::value;
    const int lane = lane_id();
    const long long out = rpC[r];
    long long room = rpC[r + 1] - out;
    warp_sort_keys<ITEMS>(key);
    if constexpr (HV) {
#pragma unroll
        for (int t = 0; t < ITEMS; ++t) sorted[32 * t + lane] = key[t];
        __syncwarp();
    }
    // heads: the first key of each column
    bool head[ITEMS];
    int pos[ITEMS];
    int cnt = 0;
#pragma unroll
    for (int t = 0; t < ITEMS; ++t) {
        unsigned before = __shfl_up_sync(kFull, key[t], 1);
        if (t > 0) {
            const unsigned last = __shfl_sync(kFull, key[t > 0 ? t - 1 : 0], 31);
            if (lane == 0) before = last;
        }
        head[t] = 32 * t + lane < np &&
                  ((t == 0 && lane == 0) || (before >> B) != (key[t] >> B));
        const unsigned m = __ballot_sync(kFull, head[t]);
        pos[t] = cnt + __popc(m & lanemask_lt());
        cnt += __popc(m);
    }
    if (rowend != nullptr) {
        if (cnt > room) {
            if (lane == 0) {
                overflow[atomicAdd(overflow_count, 1u)] = (int32_t)r;
                rowend[r] = -1;
            }
            __syncwarp();
            return;
        }
        room = cnt;
        if (lane == 0) rowend[r] = out + cnt;
    } else if (cnt != room && lane == 0) {
        atomicExch(err, (int)kDevCountMismatch);
    }
    if (out + room > cap && lane == 0) atomicExch(err, (int)kDevCapacity);
    V sum[ITEMS];
    if constexpr (HV) {
        bool more[ITEMS];
#pragma unroll
        for (int t = 0; t < ITEMS; ++t) {
            sum[t] = VOps<V>::init();
            if (head[t]) {
                const V x = vals[key[t] & kPlace];
                // the identity plus x is x, bit for bit, for (+, x)
                if constexpr (kPlain) sum[t] = x;
                else sum[t] = VOps<V>::add(sum[t], x);
            }
            more[t] = head[t];
        }
        for (int d = 1;; ++d) {
            bool any = false;
#pragma unroll
            for (int t = 0; t < ITEMS; ++t) {
                const int i = 32 * t + lane + d;
                unsigned x = 0u;
                more[t] = more[t] && i < np;
                if (more[t]) x = sorted[i];
                more[t] = more[t] && (x >> B) == (key[t] >> B);
                if (more[t]) sum[t] = VOps<V>::add(sum[t], vals[x & kPlace]);
                any = any || more[t];
            }
            if (!__any_sync(kFull, any)) break;
        }
    }
#pragma unroll
    for (int t = 0; t < ITEMS; ++t)
        if (head[t] && pos[t] < room && out + pos[t] < cap) {
            ciC[out + pos[t]] = (IT)(key[t] >> B);
            if constexpr (HV) vC[out + pos[t]] = sum[t];
        }
    __syncwarp();   // the keys and values have been read: the next row may write them
}

// --------------------------------------------------- symbolic: hash rows
// One warp per row; table of 2^LOG2T keys per warp.  Row count -> rowcnt[i].
template <class IT, int LOG2T, int WARPS>
__device__ __forceinline__ void symbolic_hash_kernel_body(
    const ProdDesc* __restrict__ D, const long long* __restrict__ rb,
                         int nprod, const int32_t* __restrict__ rows, const DevCounters* cnt,
                         int cls, int64_t* __restrict__ rowcnt, int* err,
        const long long vbid, const long long vnb) {
    using K = typename KeyT<IT>::type;
    constexpr int T = 1 << LOG2T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = lane_id();
    const int w = threadIdx.x >> 5;
    const long long nrows = (long long)cnt->class_count[cls];
    const int32_t* crow = rows + cnt->class_off[cls];
    const long long gw = (long long)vbid * WARPS + w;
    const long long nw = (long long)vnb * WARPS;
    if constexpr (LOG2T == kShortLog2T) {
        // rows of at most 32 products: no table
        for_class_rows<IT, NoVal>(D, rb, nprod, crow, gw, nrows, nw,
                                  [&](const RowCtx<IT, NoVal>& c, long long r) {
                                      short_row_symbolic<IT>(c, r, rowcnt, err);
                                  });
        return;
    }
    K* keys = reinterpret_cast<K*>(smem_raw) + (size_t)w * T;
    for (int s = lane; s < T; s += 32) keys[s] = K(-1);
    __syncwarp();
    for (long long rr = gw; rr < nrows; rr += nw) {
        const long long r = crow[rr];
        const RowCtx<IT, NoVal> c = row_ctx<IT, NoVal>(D, rb, nprod, r);
        const long long a0 = c.a0, a1 = c.a1;
        const IT* ciA = c.ciA;
        const int64_t* rpB = c.rpB;
        const IT* ciB = c.ciB;
        int count = 0;
        for (long long b = a0; b < a1; b += 32) {
            const int nb = (int)min(32LL, a1 - b);
            long long lo = 0;
            int len = 0;
            if (lane < nb) {
                long long k = (long long)ciA[b + lane];
                lo = rpB[k];
                len = (int)(rpB[k + 1] - lo);
            }
            walk_flat4(nb, lo, len, [&](const long long (&q)[4], const int (&)[4],
                                        const bool (&valid)[4]) {
                K kk[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) kk[t] = valid[t] ? (K)ciB[q[t]] : K(-1);
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    bool is_new = false;
                    if (valid[t]) hash_insert<LOG2T>(keys, kk[t], is_new, err);
                    count += __popc(__ballot_sync(kFull, is_new));
                }
            });
        }
        if (lane == 0) rowcnt[r] = count;
        for (int s = lane; s < T; s += 32) keys[s] = K(-1);
        __syncwarp();
    }
}

template <class IT, int LOG2T, int WARPS>
__global__ void __launch_bounds__(WARPS * 32)
    symbolic_hash_kernel(const ProdDesc* __restrict__ D, const long long* __restrict__ rb,
                         int nprod, const int32_t* __restrict__ rows, const DevCounters* cnt,
                         int cls, int64_t* __restrict__ rowcnt, int* err) {
    symbolic_hash_kernel_body<IT, LOG2T, WARPS>(D, rb, nprod, rows, cnt, cls, rowcnt, err,
        (long long)blockIdx.x, (long long)gridDim.x);
}

// -------------------------------------------------- symbolic: dense rows
// One block per row (dynamic row grabbing), bitmap of the product's n columns
// in shared memory (sized for the largest n of the batch).  Also writes the
// per-chunk counts chunkcnt[chunk_base + i*P + c] (chunk c covers columns
// [c*W, (c+1)*W)), which the numeric phase uses to skip empty chunks.
// MAXT / MINB: launch bounds of the instantiation (a register cap that lets
// four 256-thread or two 512-thread blocks share an SM -- for six and three it
// spills, 0.085 against 0.074 ms on 10007 vertices -- or one 1024-thread block
// for a bitmap that leaves room for only one block).
// Groups: the block may be split into `groups` equal groups of whole warps
// (named barriers 1..groups), each with its own bitmap of max_words words,
// so that several rows are in flight in one block; groups == 1 is the
// whole block.
constexpr int kMaxSymGroups = 8;

__device__ __forceinline__ void group_sync(int g, int gthreads, int groups) {
    if (groups == 1) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "r"(gthreads) : "memory");
}

// Sets the bits of the row's columns, by `nwarps` warps together (the order does
// not matter).  A entries are taken 32 at a time: by all warps while the row
// has no more than 32 per warp -- each then takes every nwarps-th piece of 256
// products -- else by one warp each.  (One warp per 32 entries whatever the row
// left the others waiting for it: rows of 17 A entries hold 16000 to 65000
// products of an R-MAT 18 square, and the pass spent 16 of 26 cycles between
// instructions at the barrier.)  Long rows of B go eight loads at a time.  One
// shared atomic per product: OR-ing the lanes' bits of a common word first (a
// segmented scan, or __match_any_sync with __reduce_or_sync) was measured 3x and
// 5x slower, testing the bit before 1.3x.
// R-MAT 18: 11.9 -> 7.2 ms; 100003 vertices, 8 per vertex: 1.02 -> 0.55 ms; 10007
// vertices 0.143 -> 0.074 ms.
template <class IT>
__device__ __forceinline__ void mark_row_columns(const RowCtx<IT, NoVal>& cx, unsigned* bm, int w,
                                                 int nwarps) {
    const int lane = lane_id();
    const IT* ciB = cx.ciB;
    const bool shared = cx.a1 - cx.a0 <= 32LL * nwarps;
    const int first = shared ? w : 0, step = shared ? nwarps : 1;
    const long long stride = shared ? 32 : 32LL * nwarps;
    for (long long b = cx.a0 + (shared ? 0 : 32LL * w); b < cx.a1; b += stride) {
        long long lo = 0;
        int len = 0;
        if (b + lane < cx.a1) {
            const long long k = (long long)cx.ciA[b + lane];
            lo = cx.rpB[k];
            len = (int)(cx.rpB[k + 1] - lo);
        }
        // rows of B of 32 entries and more, in pieces of 256
        const int pieces = len >= 32 ? (len + 255) >> 8 : 0;
        const int incl = warp_incl_scan(pieces);
        const int before = incl - pieces;
        const int total = __shfl_sync(kFull, incl, 31);
        for (int p = first; p < total; p += step) {
            // the last entry whose pieces start at or before p (one without
            // pieces starts where the next does)
            const int e = 31 - __clz(__ballot_sync(kFull, before <= p));
            const int at = (p - __shfl_sync(kFull, before, e)) << 8;
            const IT* cb = ciB + __shfl_sync(kFull, lo, e) + at + lane;
            const int left = __shfl_sync(kFull, len, e) - at;
            IT j[8];
            if (left >= 256) {
#pragma unroll
                for (int t = 0; t < 8; ++t) j[t] = cb[32 * t];
#pragma unroll
                for (int t = 0; t < 8; ++t) atomicOr(&bm[j[t] >> 5], 1u << (j[t] & 31));
            } else {
#pragma unroll
                for (int t = 0; t < 8; ++t) j[t] = 32 * t + lane < left ? cb[32 * t] : IT(-1);
#pragma unroll
                for (int t = 0; t < 8; ++t)
                    if (j[t] >= 0) atomicOr(&bm[j[t] >> 5], 1u << (j[t] & 31));
            }
        }
        // shorter ones, flattened: 128 products per step
        const int slen = len < 32 ? len : 0;
        if (__any_sync(kFull, slen > 0)) {
            const int sincl = warp_incl_scan(slen);
            const int sbefore = sincl - slen;
            const int stotal = __shfl_sync(kFull, sincl, 31);
            for (int f0 = 128 * first; f0 < stotal; f0 += 128 * step) {
                IT j[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int f = f0 + 32 * t + lane;
                    // the last entry that starts at or before f
                    int e = 0;
#pragma unroll
                    for (int d = 16; d; d >>= 1)
                        if (__shfl_sync(kFull, sbefore, e + d) <= f) e += d;
                    const long long q =
                        __shfl_sync(kFull, lo, e) + (f - __shfl_sync(kFull, sbefore, e));
                    j[t] = f < stotal ? ciB[q] : IT(-1);
                }
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    if (j[t] >= 0) atomicOr(&bm[j[t] >> 5], 1u << (j[t] & 31));
            }
        }
    }
}

template <class IT, int MAXT, int MINB>
__device__ __forceinline__ void symbolic_dense_kernel_body(const ProdDesc* __restrict__ D,
                                      const long long* __restrict__ rb, int nprod,
                                      const int32_t* __restrict__ rows, const DevCounters* cnt,
                                      int max_words, int chunk_words,
                                      int32_t* __restrict__ chunkcnt, int64_t* __restrict__ rowcnt,
                                      unsigned long long* work, int* err,
                                      unsigned* __restrict__ kept,
        const long long vbid, const long long vnb, const int groups = 1) {
    extern __shared__ unsigned bm_all[];
    __shared__ long long row_total_g[kMaxSymGroups];
    __shared__ long long cur_row_g[kMaxSymGroups];
    const int gthreads = blockDim.x / groups;
    const int g = threadIdx.x / gthreads;
    const int gt = threadIdx.x - g * gthreads;
    unsigned* bm = bm_all + (size_t)g * max_words;
    long long& row_total = row_total_g[g];
    long long& cur_row = cur_row_g[g];
    const int lane = lane_id();
    const int w = gt >> 5;
    const int nwarps = gthreads >> 5;
    unsigned long long nd = 0;
    for (int t = kClassDense0; t < kNumClasses; ++t) nd += cnt->class_count[t];
    const long long nrows = (long long)nd;
    const int32_t* drow = rows + cnt->class_off[kClassDense0];
    for (int t = gt; t < max_words; t += gthreads) bm[t] = 0u;
    if (gt == 0) row_total = 0;
    group_sync(g, gthreads, groups);
    while (true) {
        if (gt == 0) cur_row = (long long)atomicAdd(work, 1ull);
        group_sync(g, gthreads, groups);
        const long long rr = cur_row;
        if (rr >= nrows) break;
        const long long r = drow[rr];
        const RowCtx<IT, NoVal> cx = row_ctx<IT, NoVal>(D, rb, nprod, r);
        const int NW = (int)((cx.n + 31) >> 5);
        const int P = cx.P;
        if (NW > max_words) {  // n beyond the shared-memory bitmap: reported, row skipped
            if (gt == 0) atomicExch(err, (int)kDevTooWide);
            group_sync(g, gthreads, groups);
            continue;
        }
        mark_row_columns<IT>(cx, bm, w, nwarps);
        group_sync(g, gthreads, groups);
        long long part = 0;
        for (int c = w; c < P; c += nwarps) {
            const int w0 = c * chunk_words;
            const int w1 = min(NW, w0 + chunk_words);
            int s = 0;
            for (int t = w0 + lane; t < w1; t += 32) {
                const unsigned word = bm[t];
                s += __popc(word);
                if (kept) kept[rr * max_words + t] = word;
                bm[t] = 0u;
            }
            s = warp_sum(s);
            if (lane == 0) chunkcnt[cx.chunk_base + cx.i * P + c] = s;
            part += s;
        }
        if (lane == 0 && part) atomicAdd((unsigned long long*)&row_total, (unsigned long long)part);
        group_sync(g, gthreads, groups);
        if (gt == 0) {
            rowcnt[r] = row_total;
            row_total = 0;
        }
        group_sync(g, gthreads, groups);
    }
}

template <class IT, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) symbolic_dense_kernel(const ProdDesc* __restrict__ D,
                                      const long long* __restrict__ rb, int nprod,
                                      const int32_t* __restrict__ rows, const DevCounters* cnt,
                                      int max_words, int chunk_words,
                                      int32_t* __restrict__ chunkcnt, int64_t* __restrict__ rowcnt,
                                      unsigned long long* work, int* err,
                                      unsigned* __restrict__ kept) {
    symbolic_dense_kernel_body<IT, MAXT, MINB>(D, rb, nprod, rows, cnt, max_words, chunk_words,
        chunkcnt, rowcnt, work, err, kept, (long long)blockIdx.x, (long long)gridDim.x);
}

// The columns of the dense rows of a pattern from the bitmaps the symbolic
// pass kept (max_words words per dense row): a block per row, each warp a range of
// chunks; the chunks' counts give its place in C(i,:).  A lane takes four words
// and puts their bits' offsets into the warp's stage, highest first (one
// instruction of the slow pipe per bit), so that the stores to C are coalesced.
// What bounds it: instructions, the bit loops (issue 75 % active, DRAM 28 % of
// its peak); sweeping the products of every row again took as long as their
// symbolic pass.  R-MAT, 100003 vertices (233 M columns): sweep 1.82 ms, a word
// per lane and a scan for each 0.63 ms, four 0.59 ms; loading a step ahead 0.60 ms.
constexpr int kColStage = 512;   // of the 4096 columns of 128 words
template <class IT>
__global__ void __launch_bounds__(256, 8)
    dense_columns_kernel(const ProdDesc* __restrict__ D, const long long* __restrict__ rb,
                         int nprod, const int32_t* __restrict__ rows, const DevCounters* cnt,
                         const unsigned* __restrict__ kept, int max_words, int chunk_words,
                         const int32_t* __restrict__ chunkcnt, const int64_t* __restrict__ rpC,
                         long long cap, IT* __restrict__ ciC, int* err) {
    __shared__ unsigned short stage_all[8][kColStage];
    const int lane = lane_id(), w = threadIdx.x >> 5;
    unsigned short* stage = stage_all[w];
    const long long nrows = (long long)(cnt->class_off[kNumClasses] - cnt->class_off[kClassDense0]);
    const int32_t* drow = rows + cnt->class_off[kClassDense0];
    for (long long rr = blockIdx.x; rr < nrows; rr += gridDim.x) {
        const long long r = drow[rr];
        const ProdDesc& d = D[nprod > 1 ? find_prod(rb, nprod, r) : 0];
        const int P = d.P, NW = (int)((d.n + 31) >> 5);
        const int32_t* ccnt = chunkcnt + d.chunk_base + (r - d.row_base) * P;
        const unsigned* words = kept + rr * max_words;
        const long long out = rpC[r], end = rpC[r + 1];
        const int cs = (int)((long long)P * w / 8), ce = (int)((long long)P * (w + 1) / 8);
        long long before = 0, own = 0;
        for (int c = lane; c < ce; c += 32) {
            if (c < cs) before += ccnt[c];
            else own += ccnt[c];
        }
        before = warp_sum(before);
        own = warp_sum(own);
        // the row pointers are the caller's: no warp writes outside its part of them
        if (out < 0 || end > cap || out + before + own > end ||
            (w == 7 && out + before + own != end)) {
            if (lane == 0) atomicExch(err, end > cap ? (int)kDevCapacity : (int)kDevCountMismatch);
            continue;
        }
        IT* dst = ciC + out + before;
        const int t1 = min(NW, ce * chunk_words);
        for (int b = cs * chunk_words; b < t1; b += 128) {
            unsigned word[4];
            int pc = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int t = b + 4 * lane + u;
                word[u] = t < t1 ? words[t] : 0u;
                pc += __popc(word[u]);
            }
            const int incl = warp_incl_scan(pc);
            const int total = __shfl_sync(kFull, incl, 31);
            int p = incl - 1;   // the place of this lane's highest bit left
            for (int to = total; to > 0; to -= kColStage) {
                const int from = max(0, to - kColStage);
#pragma unroll
                for (int u = 3; u >= 0; --u)
                    while (word[u] && p >= from) {
                        const int bit = 31 - __clz(word[u]);
                        stage[p - from] = (unsigned short)(lane * 128 + u * 32 + bit);
                        word[u] ^= 1u << bit;
                        --p;
                    }
                __syncwarp();
                for (int x = from + lane; x < to; x += 32)
                    dst[x] = (IT)((long long)b * 32 + stage[x - from]);
                __syncwarp();
            }
            dst += total;
        }
    }
}

// ---------------------------------------------------- numeric: hash rows
template <class K, class V>
__device__ __forceinline__ void warp_bitonic_sort(K* keys, V* vals, int N) {
    const int lane = lane_id();
    for (int k = 2; k <= N; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = lane; i < N; i += 32) {
                int ixj = i ^ j;
                if (ixj > i) {
                    K ki = keys[i], kj = keys[ixj];
                    bool up = (i & k) == 0;
                    if ((ki > kj) == up) {
                        keys[i] = kj;
                        keys[ixj] = ki;
                        if constexpr (VOps<V>::has_val) {
                            V t = vals[i];
                            vals[i] = vals[ixj];
                            vals[ixj] = t;
                        }
                    }
                }
            }
            __syncwarp();
        }
    }
}

// Stable LSD radix sort of N (key, value) pairs by one warp, 8-bit digits
// over the low `bits` bits of the keys (keys are >= 0).  Ping-pongs between
// (k0, v0) and (k1, v1); returns true if the sorted pairs end in (k1, v1).
// Each pass: digit histogram, exclusive scan, then a scatter in rounds of 32
// keys in input order where lanes with equal digits take consecutive slots
// in lane order, so equal digits keep their input order.
template <class K, class V>
__device__ __forceinline__ bool warp_radix_sort(K* k0, V* v0, K* k1, V* v1, int N, int bits,
                                                int* cnt) {
    constexpr bool HV = VOps<V>::has_val;
    const int lane = lane_id();
    bool flip = false;
    for (int shift = 0; shift < bits; shift += 8) {
        K* kin = flip ? k1 : k0;
        V* vin = flip ? v1 : v0;
        K* kout = flip ? k0 : k1;
        V* vout = flip ? v0 : v1;
        for (int t = lane; t < 256; t += 32) cnt[t] = 0;
        __syncwarp();
        for (int i = lane; i < N; i += 32) atomicAdd(&cnt[(int)((kin[i] >> shift) & 255)], 1);
        __syncwarp();
        int loc[8];
        int sum = 0;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            loc[t] = cnt[lane * 8 + t];
            sum += loc[t];
        }
        int run = warp_incl_scan(sum) - sum;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            cnt[lane * 8 + t] = run;
            run += loc[t];
        }
        __syncwarp();
        for (int i0 = 0; i0 < N; i0 += 32) {
            const int i = i0 + lane;
            const bool valid = i < N;
            K kk = valid ? kin[i] : K(0);
            V vv{};
            if constexpr (HV)
                if (valid) vv = vin[i];
            const int d = valid ? (int)((kk >> shift) & 255) : 256 + lane;
            const unsigned grp = __match_any_sync(kFull, d);
            const int rank = __popc(grp & lanemask_lt());
            const int base = valid ? cnt[d] : 0;
            __syncwarp();
            if (valid) {
                kout[base + rank] = kk;
                if constexpr (HV) vout[base + rank] = vv;
                if ((grp >> lane) == 1u) cnt[d] = base + __popc(grp);  // highest lane of the group
            }
            __syncwarp();
        }
        flip = !flip;
    }
    return flip;
}

// One warp per row; table of 2^LOG2T (key, value) slots; products added in
// ascending k (ordered rounds); table compacted, sorted, written.  Rows of at
// most 128 products (bin 1) are sorted in registers instead, where their
// columns allow it.
template <class IT, class V, int LOG2T, int WARPS>
__device__ __forceinline__ void numeric_hash_kernel_body(
    const ProdDesc* __restrict__ D, const long long* __restrict__ rb,
                        int nprod, const int32_t* __restrict__ rows, const DevCounters* cnt,
                        int cls, const int64_t* __restrict__ rpC, long long cap,
                        IT* __restrict__ ciC, V* __restrict__ vC, int* err,
                        int64_t* __restrict__ rowend, int32_t* __restrict__ overflow,
                        unsigned* overflow_count,
        const long long vbid, const long long vnb) {
    using K = typename KeyT<IT>::type;
    constexpr int T = 1 << LOG2T;
    constexpr bool HV = VOps<V>::has_val;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = lane_id();
    const int w = threadIdx.x >> 5;
    if constexpr (LOG2T == kShortLog2T) {
        // rows of at most 32 products: no table
        const long long nrows = (long long)cnt->class_count[cls];
        const int32_t* crow = rows + cnt->class_off[cls];
        const long long gw = (long long)vbid * WARPS + w;
        const long long nw = (long long)vnb * WARPS;
        for_class_rows<IT, V>(D, rb, nprod, crow, gw, nrows, nw,
                              [&](const RowCtx<IT, V>& c, long long r) {
                                  short_row_numeric<IT, V>(c, r, rpC, cap, ciC, vC, err, rowend,
                                                           overflow, overflow_count);
                              });
        return;
    }
    // layout per warp: T values (if any), T keys, 256 radix counters
    constexpr size_t vbytes = HV ? sizeof(V) * T : 0;
    unsigned char* base = smem_raw + (size_t)w * (vbytes + sizeof(K) * T + 256 * sizeof(int));
    V* acc = reinterpret_cast<V*>(base);
    K* keys = reinterpret_cast<K*>(base + vbytes);
    int* rcnt_smem = reinterpret_cast<int*>(base + vbytes + sizeof(K) * T);
    // slot mode (learned sizing): rows go to predicted slots [rpC[r], rpC[r+1]);
    // a row that does not fit its slot or its table is listed for an exact re-run
    const bool slot_mode = rowend != nullptr;
    __shared__ int warp_fail[WARPS];
    int* fail = slot_mode ? &warp_fail[w] : err;
    if (lane == 0) warp_fail[w] = 0;
    __syncwarp();
    for (int s = lane; s < T; s += 32) {
        keys[s] = K(-1);
        if constexpr (HV) acc[s] = VOps<V>::init();
    }
    __syncwarp();
    const long long nrows = (long long)cnt->class_count[cls];
    const int32_t* crow = rows + cnt->class_off[cls];
    const long long gw = (long long)vbid * WARPS + w;
    const long long nw = (long long)vnb * WARPS;
    bool clean = true;   // the table is empty
    for (long long rr = gw; rr < nrows; rr += nw) {
        const long long r = crow[rr];
        const RowCtx<IT, V> c = row_ctx<IT, V>(D, rb, nprod, r);
        if constexpr (LOG2T == 8) {
            // with the learned predictor a row of this bin may have more
            // products: it takes the table
            if (sortable_columns<4>(c.n)) {
                unsigned key[4];
                unsigned* sorted = reinterpret_cast<unsigned*>(keys);
                const int np = sorted_row_gather<IT, V, 4>(c, key, acc);
                clean = false;
                if (np >= 0) {
                    __syncwarp();
                    if (np <= 64) {
                        // the same keys with the place in six bits
                        unsigned k2[2] = {key[0], key[1]};
#pragma unroll
                        for (int t = 0; t < 2; ++t)
                            if (k2[t] != 0xffffffffu) k2[t] = (k2[t] >> 7) << 6 | (k2[t] & 63u);
                        sorted_row_numeric<IT, V, 2>(k2, np, r, acc, sorted, rpC, cap, ciC, vC,
                                                     err, rowend, overflow, overflow_count);
                    } else {
                        sorted_row_numeric<IT, V, 4>(key, np, r, acc, sorted, rpC, cap, ciC, vC,
                                                     err, rowend, overflow, overflow_count);
                    }
                    continue;
                }
                __syncwarp();
            }
            if (!clean) {
                for (int s = lane; s < T; s += 32) {
                    keys[s] = K(-1);
                    if constexpr (HV) acc[s] = VOps<V>::init();
                }
                __syncwarp();
                clean = true;
            }
        }
        const long long a0 = c.a0, a1 = c.a1;
        const IT* ciA = c.ciA;
        const V* vA = c.vA;
        const int64_t* rpB = c.rpB;
        const IT* ciB = c.ciB;
        const V* vB = c.vB;
        // A row of at most 32 A entries has its one batch loaded here, once.
        // If its products hardly repeat a column (nnz(C(i,:)) >= 3/4 of its
        // flops, known exactly outside slot mode) and fit half the table, it
        // is expanded, sorted and compressed instead of hashed: products go
        // to the table's lower half in ascending k, a stable radix sort by
        // column keeps that order among equal columns, and each run of equal
        // columns is reduced from the identity in that order, as the hash
        // path would.
        bool pre = false;
        long long lo_p = 0;
        int len_p = 0;
        V a_p = VOps<V>::init();
        if constexpr (LOG2T >= 10) {
            if (!slot_mode && a1 > a0 && a1 - a0 <= 32) {
                const int nb = (int)(a1 - a0);
                if (lane < nb) {
                    const long long k = (long long)ciA[a0 + lane];
                    lo_p = rpB[k];
                    len_p = (int)(rpB[k + 1] - lo_p);
                    a_p = load_val(vA, a0 + lane);
                }
                pre = true;
                const long long fl = warp_sum((long long)len_p);
                const long long nz = rpC[r + 1] - rpC[r];
                if (fl <= T / 2 && 4 * nz >= 3 * fl) {
                    int nf = 0;
                    walk_batch4(nb, lo_p, len_p, [&](const long long (&q)[4], const int (&e)[4],
                                                     const bool (&vl)[4], bool) {
                        K key[4];
                        V bq[4];
                        V ae[4];
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            ae[t] = shfl_val(a_p, e[t]);
                            key[t] = K(0);
                            bq[t] = V{};
                            if (vl[t]) {
                                key[t] = (K)ciB[q[t]];
                                bq[t] = load_val(vB, q[t]);
                            }
                        }
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            // the valid lanes of a round are a prefix of the warp
                            if (vl[t]) {
                                keys[nf + lane] = key[t];
                                if constexpr (HV) acc[nf + lane] = VOps<V>::mul(ae[t], bq[t]);
                            }
                            nf += __popc(__ballot_sync(kFull, vl[t]));
                        }
                    });
                    __syncwarp();
                    const int bits = c.n > 1 ? 64 - __clzll((unsigned long long)(c.n - 1)) : 1;
                    const bool up = warp_radix_sort<K, V>(keys, acc, keys + T / 2, acc + T / 2, nf,
                                                          bits, rcnt_smem);
                    const K* sk = up ? keys + T / 2 : keys;
                    const V* sv = up ? acc + T / 2 : acc;
                    const long long out = rpC[r];
                    int outp = 0;
                    for (int i0 = 0; i0 < nf; i0 += 32) {
                        const int i = i0 + lane;
                        const bool in = i < nf;
                        const K kk = in ? sk[i] : K(0);
                        const bool start = in && (i == 0 || sk[i - 1] != kk);
                        const unsigned sm = __ballot_sync(kFull, start);
                        if (start) {
                            V sum = VOps<V>::init();
                            if constexpr (HV) {
                                sum = VOps<V>::add(sum, sv[i]);
                                for (int j = i + 1; j < nf && sk[j] == kk; ++j)
                                    sum = VOps<V>::add(sum, sv[j]);
                            }
                            const long long pq = out + outp + __popc(sm & lanemask_lt());
                            if (pq < cap) {
                                ciC[pq] = (IT)kk;
                                if constexpr (HV) vC[pq] = sum;
                            }
                        }
                        outp += __popc(sm);
                    }
                    if (lane == 0 && (long long)outp != nz) atomicExch(err, (int)kDevCountMismatch);
                    if (lane == 0 && out + outp > cap) atomicExch(err, (int)kDevCapacity);
                    __syncwarp();
                    // both halves back to the empty table
                    for (int t = lane; t < nf; t += 32) {
                        keys[t] = K(-1);
                        keys[T / 2 + t] = K(-1);
                        if constexpr (HV) {
                            acc[t] = VOps<V>::init();
                            acc[T / 2 + t] = VOps<V>::init();
                        }
                    }
                    __syncwarp();
                    continue;
                }
            }
        }
        for (long long b = a0; b < a1; b += 32) {
            const int nb = (int)min(32LL, a1 - b);
            long long lo = 0;
            int len = 0;
            V a = VOps<V>::init();
            if (pre) {  // the row's single batch, loaded above
                lo = lo_p;
                len = len_p;
                a = a_p;
            } else if (lane < nb) {
                long long k = (long long)ciA[b + lane];
                lo = rpB[k];
                len = (int)(rpB[k + 1] - lo);
                a = load_val(vA, b + lane);
            }
            // four rounds per step: their loads are issued together, then
            // the rounds are inserted and accumulated in order
            walk_batch4(nb, lo, len, [&](const long long (&q)[4], const int (&e)[4],
                                         const bool (&vl)[4], bool ordered) {
                K key[4];
                V bq[4];
                V ae[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    ae[t] = shfl_val(a, e[t]);
                    key[t] = K(-1);
                    bq[t] = V{};
                    if (vl[t]) {
                        key[t] = (K)ciB[q[t]];
                        bq[t] = load_val(vB, q[t]);
                    }
                }
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    int slot = -1;
                    V v{};
                    if (vl[t]) {
                        bool is_new;
                        slot = hash_insert<LOG2T>(keys, key[t], is_new, fail);
                        v = VOps<V>::mul(ae[t], bq[t]);
                    }
                    const bool valid = vl[t] && slot >= 0;
                    if (ordered) ordered_add(acc, slot, valid, v);
                    else plain_add(acc, slot, valid, v);
                }
            });
        }
        // compact occupied slots to the front (ascending slot order)
        const long long out = rpC[r];
        int rcnt = (int)(rpC[r + 1] - out);
        int pos = 0;
        for (int s0 = 0; s0 < T; s0 += 32) {
            K kk = keys[s0 + lane];
            V vv{};
            if constexpr (HV) vv = acc[s0 + lane];
            bool occ = kk != K(-1);
            unsigned msk = __ballot_sync(kFull, occ);
            __syncwarp();
            int p = pos + __popc(msk & lanemask_lt());
            if (occ) {
                keys[p] = kk;
                if constexpr (HV) acc[p] = vv;
            }
            pos += __popc(msk);
            __syncwarp();
        }
        if (slot_mode) {
            __syncwarp();
            const bool bad = warp_fail[w] != 0 || pos > rcnt;
            if (bad) {
                if (lane == 0) {
                    overflow[atomicAdd(overflow_count, 1u)] = (int32_t)r;
                    rowend[r] = -1;
                    warp_fail[w] = 0;
                }
                for (int sl = lane; sl < T; sl += 32) {
                    keys[sl] = K(-1);
                    if constexpr (HV) acc[sl] = VOps<V>::init();
                }
                __syncwarp();
                continue;
            }
            rcnt = pos;
            if (lane == 0) rowend[r] = out + pos;
        } else if (pos != rcnt && lane == 0) {
            atomicExch(err, (int)kDevCountMismatch);
        }
        if (out + rcnt > cap && lane == 0) atomicExch(err, (int)kDevCapacity);
        const K* sk = keys;
        const V* sv = acc;
        if (pos <= 64) {
            int N = 1;
            while (N < pos) N <<= 1;
            const K kmax = sizeof(K) == 4 ? (K)0x7fffffff : (K)0x7fffffffffffffffLL;
            for (int s = pos + lane; s < N; s += 32) keys[s] = kmax;
            __syncwarp();
            warp_bitonic_sort<K, V>(keys, acc, N);
        } else {
            // pos <= T/2: the upper half of the table is the second buffer
            const int bits = c.n > 1 ? 64 - __clzll((unsigned long long)(c.n - 1)) : 1;
            const bool in_upper = warp_radix_sort<K, V>(keys, acc, keys + T / 2, acc + T / 2, pos,
                                                        bits, rcnt_smem);
            if (in_upper) {
                sk = keys + T / 2;
                sv = acc + T / 2;
            }
        }
        const int lim = (int)max(0LL, min((long long)min(pos, rcnt), cap - out));
        for (int t = lane; t < lim; t += 32) {
            ciC[out + t] = (IT)sk[t];
            if constexpr (HV) vC[out + t] = sv[t];
        }
        __syncwarp();
        for (int s = lane; s < T; s += 32) {
            keys[s] = K(-1);
            if constexpr (HV) acc[s] = VOps<V>::init();
        }
        __syncwarp();
    }
}

template <class IT, class V, int LOG2T, int WARPS>
__global__ void __launch_bounds__(WARPS * 32)
    numeric_hash_kernel(const ProdDesc* __restrict__ D, const long long* __restrict__ rb,
                        int nprod, const int32_t* __restrict__ rows, const DevCounters* cnt,
                        int cls, const int64_t* __restrict__ rpC, long long cap,
                        IT* __restrict__ ciC, V* __restrict__ vC, int* err,
                        int64_t* __restrict__ rowend, int32_t* __restrict__ overflow,
                        unsigned* overflow_count) {
    numeric_hash_kernel_body<IT, V, LOG2T, WARPS>(D, rb, nprod, rows, cnt, cls, rpC, cap, ciC,
        vC, err, rowend, overflow, overflow_count, (long long)blockIdx.x, (long long)gridDim.x);
}

// One run of a batch of A entries whose products are flattened: product f of
// the run sits at B position off + f, and is scaled by a = A(i,k).
template <class V>
struct __align__(16) DenseRun {
    long long off;
    V a;
};

// ------------------------- rows of 129 to 1024 products, ranked by a bitmap
// Hash bins 2 (counts, and slots of predicted size) and 3 in products of at most
// rank_max_n columns.  A block of four
// warps takes a row; product f of the row (ascending k) sits in warp (f / 32) %
// 4, lane f % 32, item f / 128.  The products set the bits of their columns;
// the set bits before a column are its place in C(i,:), so nothing is hashed or
// sorted.  The first product of every place (the smallest f, by atomicMin)
// stores its value; the others, few in a sparse row, are listed in ascending f
// and added by one warp in that order.
// What bounds it: instructions and shared memory (numeric float32: issue 57 %, L1
// 74 %), at 24 to 36 warps per SM.  A warp with a table
// per row (25 KB for float64) held 12 warps and took 9.7 instructions per
// product: 64 uneven Erdos-Renyi products in float32 (up to 65536 columns),
// rows of 513 to 1024 products 6.25 -> 2.34 ms, their counts 1.45 -> 0.91 ms.
constexpr int kRankWarps = 4;
constexpr int kRankItems = 8;
constexpr int kRankMost = 32 * kRankWarps * kRankItems;   // products of a row
static_assert(kRankMost >= hash_bin_flops(kNumHashBins - 1), "a hash row fits");
// Most columns for which the bitmap beats the table, by bin and pass: clearing
// and counting it costs the same whatever the row holds.
__host__ __device__ constexpr long long rank_max_n(int bin, bool count) {
    return bin == 3 ? 262144 : bin == 2 ? (count ? 16384 : 32768) : 0;
}

// Words of the bitmap of n columns: each warp takes whole groups of 128.
__host__ __device__ constexpr int rank_words(long long n) {
    return (int)((n + 128 * 32 * kRankWarps - 1) / (128 * 32 * kRankWarps)) * 128 * kRankWarps;
}

// Shared memory: the column map (bits, then the set bits before every word;
// its room is the list of later products afterwards), places' first products
// and then columns, accumulators, and a table of runs per warp.
template <class V>
struct RankSmem {
    static constexpr size_t kList = kRankMost * (sizeof(int) + (VOps<V>::has_val ? sizeof(V) : 0));
    size_t before, tag, acc, runs, total;
    __host__ __device__ explicit RankSmem(long long n, bool count) {
        before = (size_t)rank_words(n) * sizeof(unsigned);
        const size_t map = before + (count ? 0 : (size_t)rank_words(n) * sizeof(unsigned short));
        tag = ((count || map > kList ? map : kList) + 15) / 16 * 16;
        acc = tag + (count ? 0 : kRankMost * sizeof(unsigned));
        runs = acc + (!count && VOps<V>::has_val ? kRankMost * sizeof(V) : 0);
        total = runs + kRankWarps * 32 * sizeof(DenseRun<V>);
    }
};

// Columns (-1: none) and values of this lane's products of the row.
template <class IT, class V, bool VALS>
__device__ __forceinline__ void rank_gather(const RowCtx<IT, V>& c, int w, int (&col)[kRankItems],
                                            V (&v)[kRankItems], DenseRun<V>* runs) {
    const int lane = lane_id();
#pragma unroll
    for (int t = 0; t < kRankItems; ++t) {
        col[t] = -1;
        v[t] = VOps<V>::init();
    }
    int have = 0;
    for (long long b = c.a0; b < c.a1; b += 32) {
        const int nb = (int)min(32LL, c.a1 - b);
        long long lo = 0;
        int len = 0;
        DenseRun<V> run{};
        if (lane < nb) {
            const long long k = (long long)c.ciA[b + lane];
            lo = c.rpB[k];
            len = (int)min(c.rpB[k + 1] - lo, (long long)kRankMost);
            if constexpr (VALS) run.a = load_val(c.vA, b + lane);
        }
        const int incl = warp_incl_scan(len);
        const int tot = min(__shfl_sync(kFull, incl, 31), kRankMost - have);
        if (tot <= 0) continue;
        const int start = have + incl - len;
        const unsigned some = __ballot_sync(kFull, len > 0);
        run.off = lo - start;
        __syncwarp();   // the table's last use is over
        if (len > 0) runs[__popc(some & lanemask_lt())] = run;
        __syncwarp();
#pragma unroll
        for (int t = 0; t < kRankItems; ++t) {
            const int w0 = 32 * (kRankWarps * t + w);
            if (w0 >= have + tot || w0 + 32 <= have) continue;
            // the run of product f: the runs that start at or before it
            const unsigned M = __reduce_or_sync(
                kFull, len > 0 && start >= w0 && start < w0 + 32 ? 1u << (start - w0) : 0u);
            const int e = __popc(__ballot_sync(kFull, len > 0 && start < w0)) +
                          __popc(M & lanemask_le()) - 1;
            const int f = w0 + lane;
            if (f >= have && f < have + tot) {
                const DenseRun<V> x = runs[e];
                const long long q = x.off + f;
                col[t] = (int)c.ciB[q];
                if constexpr (VALS) v[t] = VOps<V>::mul(x.a, load_val(c.vB, q));
            }
        }
        have += tot;
    }
}

// Set bits before every word of the map and their total; warp w owns the words
// [w, w + 1) * nwords / 4, four per lane and step.  Two barriers; the last one
// covers the words' counts too.
__device__ __forceinline__ int rank_prefix(const unsigned* bits, unsigned short* before, int nwords,
                                           int w, int* part) {
    const int lane = lane_id();
    const int per = nwords / kRankWarps;
    const uint4* b4 = reinterpret_cast<const uint4*>(bits + w * per);
    ushort4* p4 = reinterpret_cast<ushort4*>(before + w * per);
    int sum = 0;
    for (int t = lane; t < per / 4; t += 32) {
        const uint4 x = b4[t];
        sum += __popc(x.x) + __popc(x.y) + __popc(x.z) + __popc(x.w);
    }
    sum = warp_sum(sum);
    if (lane == 0) part[w] = sum;
    __syncthreads();
    int base = 0, total = 0;
#pragma unroll
    for (int u = 0; u < kRankWarps; ++u) {
        base += u < w ? part[u] : 0;
        total += part[u];
    }
    for (int t = lane; t < per / 4; t += 32) {
        const uint4 x = b4[t];
        const int p0 = __popc(x.x), p1 = p0 + __popc(x.y), p2 = p1 + __popc(x.z),
                  p3 = p2 + __popc(x.w);
        const int incl = warp_incl_scan(p3);
        const int at = base + incl - p3;
        p4[t] = make_ushort4((unsigned short)at, (unsigned short)(at + p0),
                             (unsigned short)(at + p1), (unsigned short)(at + p2));
        base += __shfl_sync(kFull, incl, 31);
    }
    __syncthreads();
    return total;
}

__device__ __forceinline__ void rank_clear(unsigned* bits, int nwords) {
    uint4* b4 = reinterpret_cast<uint4*>(bits);
    for (int t = threadIdx.x; t < nwords / 4; t += blockDim.x) b4[t] = make_uint4(0u, 0u, 0u, 0u);
}

template <class IT>
__global__ void __launch_bounds__(32 * kRankWarps)
    symbolic_rank_kernel(const ProdDesc* __restrict__ D, const long long* __restrict__ rb,
                         int nprod, const int32_t* __restrict__ rows, const DevCounters* cnt,
                         int cls, long long max_n, int64_t* __restrict__ rowcnt) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int total;
    const RankSmem<NoVal> L(max_n, true);
    unsigned* bits = reinterpret_cast<unsigned*>(smem_raw);
    const int lane = lane_id(), w = threadIdx.x >> 5;
    DenseRun<NoVal>* runs = reinterpret_cast<DenseRun<NoVal>*>(smem_raw + L.runs) + 32 * w;
    rank_clear(bits, rank_words(max_n));
    if (threadIdx.x == 0) total = 0;
    __syncthreads();
    const long long nrows = (long long)cnt->class_count[cls];
    const int32_t* crow = rows + cnt->class_off[cls];
    for (long long rr = blockIdx.x; rr < nrows; rr += gridDim.x) {
        const long long r = crow[rr];
        const RowCtx<IT, NoVal> c = row_ctx<IT, NoVal>(D, rb, nprod, r);
        int col[kRankItems];
        NoVal v[kRankItems];
        rank_gather<IT, NoVal, false>(c, w, col, v, runs);
#pragma unroll
        for (int t = 0; t < kRankItems; ++t)
            if (col[t] >= 0) atomicOr(&bits[col[t] >> 5], 1u << (col[t] & 31));
        __syncthreads();
        int sum = 0;
        uint4* b4 = reinterpret_cast<uint4*>(bits);
        for (int t = threadIdx.x; t < rank_words(c.n) / 4; t += blockDim.x) {
            const uint4 x = b4[t];
            sum += __popc(x.x) + __popc(x.y) + __popc(x.z) + __popc(x.w);
            b4[t] = make_uint4(0u, 0u, 0u, 0u);
        }
        sum = warp_sum(sum);
        if (lane == 0 && sum) atomicAdd(&total, sum);
        __syncthreads();
        if (threadIdx.x == 0) {
            rowcnt[r] = total;
            total = 0;
        }
    }
}

template <class IT, class V>
__global__ void __launch_bounds__(32 * kRankWarps)
    numeric_rank_kernel(const ProdDesc* __restrict__ D, const long long* __restrict__ rb,
                        int nprod, const int32_t* __restrict__ rows, const DevCounters* cnt,
                        int cls, long long max_n, const int64_t* __restrict__ rpC, long long cap,
                        IT* __restrict__ ciC, V* __restrict__ vC, int* err,
                        int64_t* __restrict__ rowend, int32_t* __restrict__ overflow,
                        unsigned* overflow_count) {
    constexpr bool HV = VOps<V>::has_val;
    constexpr bool kPlain = std::is_same<V, double>::value || std::is_same<V, float>::value ||
                            std::is_same<V, int64_t>::value;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int part[32];
    const RankSmem<V> L(max_n, false);
    unsigned* bits = reinterpret_cast<unsigned*>(smem_raw);
    unsigned short* before = reinterpret_cast<unsigned short*>(smem_raw + L.before);
    V* list_v = reinterpret_cast<V*>(smem_raw);
    int* list_s = reinterpret_cast<int*>(smem_raw + (HV ? kRankMost * sizeof(V) : 0));
    unsigned* tag = reinterpret_cast<unsigned*>(smem_raw + L.tag);
    V* acc = reinterpret_cast<V*>(smem_raw + L.acc);
    const int lane = lane_id(), w = threadIdx.x >> 5;
    DenseRun<V>* runs = reinterpret_cast<DenseRun<V>*>(smem_raw + L.runs) + 32 * w;
    rank_clear(bits, rank_words(max_n));
    for (int t = threadIdx.x; t < kRankMost; t += blockDim.x) tag[t] = 0xffffffffu;
    __syncthreads();
    const long long nrows = (long long)cnt->class_count[cls];
    const int32_t* crow = rows + cnt->class_off[cls];
    for (long long rr = blockIdx.x; rr < nrows; rr += gridDim.x) {
        const long long r = crow[rr];
        const RowCtx<IT, V> c = row_ctx<IT, V>(D, rb, nprod, r);
        const long long out = rpC[r];
        const long long room = rpC[r + 1] - out;
        int col[kRankItems];
        V v[kRankItems];
        rank_gather<IT, V, HV>(c, w, col, v, runs);
#pragma unroll
        for (int t = 0; t < kRankItems; ++t)
            if (col[t] >= 0) atomicOr(&bits[col[t] >> 5], 1u << (col[t] & 31));
        __syncthreads();
        int nwords = rank_words(c.n);
        const int total = rank_prefix(bits, before, nwords, w, part);
        // slot mode: a row that outgrows its slot is listed for an exact re-run
        bool write = true;
        if (rowend != nullptr) {
            write = total <= room;
            if (threadIdx.x == 0) {
                if (!write) overflow[atomicAdd(overflow_count, 1u)] = (int32_t)r;
                rowend[r] = write ? out + total : -1;
            }
        } else if (threadIdx.x == 0) {
            if (total != room) atomicExch(err, (int)kDevCountMismatch);
            if (out + room > cap) atomicExch(err, (int)kDevCapacity);
        }
        if constexpr (HV) {
            int slot[kRankItems];
#pragma unroll
            for (int t = 0; t < kRankItems; ++t) {
                slot[t] = -1;
                if (col[t] >= 0) {
                    slot[t] = before[col[t] >> 5] +
                              __popc(bits[col[t] >> 5] & ~(0xffffffffu << (col[t] & 31)));
                    atomicMin(&tag[slot[t]], (unsigned)(32 * (kRankWarps * t + w) + lane));
                }
            }
            __syncthreads();
            bool later[kRankItems];   // not the first product of its place
            bool any = false;
#pragma unroll
            for (int t = 0; t < kRankItems; ++t) {
                later[t] = slot[t] >= 0 &&
                           tag[slot[t]] != (unsigned)(32 * (kRankWarps * t + w) + lane);
                any = any || later[t];
            }
            any = __syncthreads_or(any);
#pragma unroll
            for (int t = 0; t < kRankItems; ++t)
                if (slot[t] >= 0 && !later[t]) {
                    tag[slot[t]] = (unsigned)col[t];
                    // the identity plus x is x, bit for bit, for (+, x)
                    if constexpr (kPlain) acc[slot[t]] = v[t];
                    else acc[slot[t]] = VOps<V>::add(VOps<V>::init(), v[t]);
                }
            if (any) {
                nwords = rank_words(max_n);   // the list may lie over all of the bits
                // item t of warp w comes t * 4 + w-th
                static_assert(kRankItems * kRankWarps == 32, "a lane per group of products");
#pragma unroll
                for (int t = 0; t < kRankItems; ++t) {
                    const unsigned m = __ballot_sync(kFull, later[t]);
                    if (lane == 0) part[kRankWarps * t + w] = __popc(m);
                }
                __syncthreads();
                const int k = part[lane];
                const int incl = warp_incl_scan(k);
                const int nlist = __shfl_sync(kFull, incl, 31);
#pragma unroll
                for (int t = 0; t < kRankItems; ++t) {
                    const int at = __shfl_sync(kFull, incl - k, kRankWarps * t + w);
                    const unsigned m = __ballot_sync(kFull, later[t]);
                    if (later[t]) {
                        list_s[at + __popc(m & lanemask_lt())] = slot[t];
                        list_v[at + __popc(m & lanemask_lt())] = v[t];
                    }
                }
                __syncthreads();
                if (w == 0)
                    for (int x0 = 0; x0 < nlist; x0 += 32) {
                        const bool valid = x0 + lane < nlist;
                        ordered_add(acc, valid ? list_s[x0 + lane] : 0, valid,
                                    valid ? list_v[x0 + lane] : VOps<V>::init());
                    }
            }
            __syncthreads();
        } else {
            // the columns of the set bits, in order
            for (int t = threadIdx.x; t < nwords; t += blockDim.x) {
                unsigned p = before[t];
                for (unsigned word = bits[t]; word; word &= word - 1u)
                    tag[p++] = (unsigned)(32 * t + __ffs(word) - 1);
            }
            __syncthreads();
        }
        for (int x = threadIdx.x; x < total; x += blockDim.x) {
            if (write && x < room && out + x < cap) {
                ciC[out + x] = (IT)tag[x];
                if constexpr (HV) vC[out + x] = acc[x];
            }
            tag[x] = 0xffffffffu;
        }
        rank_clear(bits, nwords);
        __syncthreads();
    }
}

// ------------------------------ rows of 129 to 512 products, sorted by a warp
// Hash bin 2 outside slot mode.  As for the shorter rows, the products' (column,
// place) keys are sorted in registers and each run of equal columns is added up
// by the lane of its first key, in ascending place; eight or sixteen keys per
// lane.  Nine bits hold the place, so columns must be below 2^23.
// What bounds it: instructions (about two of sorting per product) and the
// gathers of the values, at 32 warps per SM where the table in float64 held 16.
// Against the table and the bitmap, Erdos-Renyi squares of 16 per column,
// numeric in us, float64 and float32: 8192 columns bitmap 42 and 39, sorted 34
// and 36; 32768 columns bitmap 160 and 143, sorted 114 and 108; 65536 columns
// table 358 and 288, sorted 220 and 213; 262144 columns table 1581 and 1248,
// sorted 925 and 844.  64 uneven products in float32: 2550 -> 2130.
constexpr int kSort9Bits = 9;
constexpr int kSort9Most = 1 << kSort9Bits;
constexpr int kSort9Warps = 8;
constexpr long long kSort9MaxN = 1LL << (32 - kSort9Bits);

// Per warp: values by place, sorted keys (a word of padding per lane), runs.
template <class V>
constexpr size_t sort9_warp_bytes() {
    return (VOps<V>::has_val ? kSort9Most * sizeof(V) : 0) + (kSort9Most + 32) * sizeof(unsigned) +
           32 * sizeof(DenseRun<V>);
}

// Ascending sort of 32 * ITEMS keys, key lane * ITEMS + t in item t: a bitonic
// network whose merges begin with a mirrored exchange, so every exchange puts
// the smaller key first and those within a lane are a min and a max.  Fifteen
// levels of exchanges between lanes, whatever ITEMS is.
template <int ITEMS>
__device__ __forceinline__ void warp_sort_blocked(unsigned (&key)[ITEMS]) {
    const int lane = lane_id();
    auto within = [&](int t, int o) {
        const unsigned x = min(key[t], key[o]), y = max(key[t], key[o]);
        key[t] = x;
        key[o] = y;
    };
#pragma unroll
    for (int k = 2; k <= 32 * ITEMS; k <<= 1) {
        if (k <= ITEMS) {
#pragma unroll
            for (int t = 0; t < ITEMS; ++t)
                if ((t ^ (k - 1)) > t) within(t, t ^ (k - 1));
        } else {
            const int m = k / ITEMS - 1;
            const bool lower = (lane & (k / ITEMS / 2)) == 0;
#pragma unroll
            for (int t = 0; t < ITEMS / 2; ++t) {
                const int o = ITEMS - 1 - t;
                const unsigned x = __shfl_xor_sync(kFull, key[o], m);
                const unsigned y = __shfl_xor_sync(kFull, key[t], m);
                key[t] = lower ? min(key[t], x) : max(key[t], x);
                key[o] = lower ? min(key[o], y) : max(key[o], y);
            }
        }
#pragma unroll
        for (int j = k >> 2; j > 0; j >>= 1) {
            if (j >= ITEMS) {
                const bool lower = (lane & (j / ITEMS)) == 0;
#pragma unroll
                for (int t = 0; t < ITEMS; ++t) {
                    const unsigned y = __shfl_xor_sync(kFull, key[t], j / ITEMS);
                    key[t] = lower ? min(key[t], y) : max(key[t], y);
                }
            } else {
#pragma unroll
                for (int t = 0; t < ITEMS; ++t)
                    if ((t ^ j) > t) within(t, t ^ j);
            }
        }
    }
}

// Sorts the first 32 * ITEMS keys and leaves key i in sorted[i + i / ITEMS]
// (no bank conflicts on the way in).
template <int ITEMS, int N>
__device__ __forceinline__ void sort9_store(const unsigned (&key)[N], unsigned* sorted) {
    unsigned k[ITEMS];
#pragma unroll
    for (int t = 0; t < ITEMS; ++t) k[t] = key[t];
    warp_sort_blocked<ITEMS>(k);
#pragma unroll
    for (int t = 0; t < ITEMS; ++t) sorted[lane_id() * (ITEMS + 1) + t] = k[t];
}

template <class IT, class V>
__global__ void __launch_bounds__(32 * kSort9Warps)
    numeric_sort_kernel(const ProdDesc* __restrict__ D, const long long* __restrict__ rb,
                        int nprod, const int32_t* __restrict__ rows, const DevCounters* cnt,
                        int cls, const int64_t* __restrict__ rpC, long long cap,
                        IT* __restrict__ ciC, V* __restrict__ vC, int* err) {
    constexpr bool HV = VOps<V>::has_val;
    constexpr bool kPlain = std::is_same<V, double>::value || std::is_same<V, float>::value ||
                            std::is_same<V, int64_t>::value;
    constexpr int B = kSort9Bits;
    constexpr int N = kSort9Most / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = lane_id(), w = threadIdx.x >> 5;
    unsigned char* base = smem_raw + w * sort9_warp_bytes<V>();
    DenseRun<V>* runs = reinterpret_cast<DenseRun<V>*>(base);
    V* vals = reinterpret_cast<V*>(base + 32 * sizeof(DenseRun<V>));
    unsigned* sorted = reinterpret_cast<unsigned*>(base + 32 * sizeof(DenseRun<V>) +
                                                   (HV ? kSort9Most * sizeof(V) : 0));
    const long long nrows = (long long)cnt->class_count[cls];
    const int32_t* crow = rows + cnt->class_off[cls];
    for (long long rr = (long long)blockIdx.x * kSort9Warps + w; rr < nrows;
         rr += (long long)gridDim.x * kSort9Warps) {
        const long long r = crow[rr];
        const RowCtx<IT, V> c = row_ctx<IT, V>(D, rb, nprod, r);
        const long long out = rpC[r];
        const long long room = rpC[r + 1] - out;
        unsigned key[N];
#pragma unroll
        for (int t = 0; t < N; ++t) key[t] = 0xffffffffu;
        int np = 0;
        for (long long b = c.a0; b < c.a1; b += 32) {
            const int nb = (int)min(32LL, c.a1 - b);
            long long lo = 0;
            int len = 0;
            DenseRun<V> run{};
            if (lane < nb) {
                const long long k = (long long)c.ciA[b + lane];
                lo = c.rpB[k];
                len = (int)min(c.rpB[k + 1] - lo, (long long)kSort9Most);
                if constexpr (HV) run.a = load_val(c.vA, b + lane);
            }
            const int incl = warp_incl_scan(len);
            const int tot = min(__shfl_sync(kFull, incl, 31), kSort9Most - np);
            if (tot <= 0) continue;
            const int start = np + incl - len;
            const unsigned some = __ballot_sync(kFull, len > 0);
            run.off = lo - start;
            __syncwarp();   // the table's last use is over
            if (len > 0) runs[__popc(some & lanemask_lt())] = run;
            __syncwarp();
#pragma unroll
            for (int t = 0; t < N; ++t) {
                if (32 * t >= np + tot || 32 * t + 32 <= np) continue;
                // the run of product f: the runs that start at or before it
                const unsigned M = __reduce_or_sync(
                    kFull,
                    len > 0 && start >= 32 * t && start < 32 * t + 32 ? 1u << (start - 32 * t) : 0u);
                const int e = __popc(__ballot_sync(kFull, len > 0 && start < 32 * t)) +
                              __popc(M & lanemask_le()) - 1;
                const int f = 32 * t + lane;
                if (f >= np && f < np + tot) {
                    const DenseRun<V> x = runs[e];
                    const long long q = x.off + f;
                    key[t] = (unsigned)c.ciB[q] << B | (unsigned)f;
                    if constexpr (HV) vals[f] = VOps<V>::mul(x.a, load_val(c.vB, q));
                }
            }
            np += tot;
        }
        const int sh = np <= 256 ? 3 : 4;   // log2 of the keys per lane
        if (np <= 256) sort9_store<8>(key, sorted);
        else sort9_store<16>(key, sorted);
        __syncwarp();
        int count = 0;
        for (int t0 = 0; t0 < np; t0 += 128) {
            unsigned x[4];
            V sum[4];
            int pos[4];
            bool more[4];
            unsigned heads = 0u;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = t0 + 32 * u + lane;
                bool head = false;
                x[u] = 0u;
                if (i < np) {
                    x[u] = sorted[i + (i >> sh)];
                    head = i == 0 || sorted[i - 1 + ((i - 1) >> sh)] >> B != x[u] >> B;
                }
                const unsigned m = __ballot_sync(kFull, head);
                pos[u] = count + __popc(m & lanemask_lt());
                count += __popc(m);
                heads |= head ? 1u << u : 0u;
                more[u] = head;
                sum[u] = VOps<V>::init();
                if constexpr (HV) {
                    if (head) {
                        const V v = vals[x[u] & (kSort9Most - 1)];
                        // the identity plus v is v, bit for bit, for (+, x)
                        if constexpr (kPlain) sum[u] = v;
                        else sum[u] = VOps<V>::add(sum[u], v);
                    }
                }
            }
            if constexpr (HV) {
                for (int d = 1;; ++d) {
                    bool any = false;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int i = t0 + 32 * u + lane + d;
                        unsigned y = 0u;
                        more[u] = more[u] && i < np;
                        if (more[u]) y = sorted[i + (i >> sh)];
                        more[u] = more[u] && y >> B == x[u] >> B;
                        if (more[u]) sum[u] = VOps<V>::add(sum[u], vals[y & (kSort9Most - 1)]);
                        any = any || more[u];
                    }
                    if (!__any_sync(kFull, any)) break;
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if ((heads >> u & 1u) && pos[u] < room && out + pos[u] < cap) {
                    ciC[out + pos[u]] = (IT)(x[u] >> B);
                    if constexpr (HV) vC[out + pos[u]] = sum[u];
                }
        }
        if (lane == 0) {
            if (count != room) atomicExch(err, (int)kDevCountMismatch);
            if (out + room > cap) atomicExch(err, (int)kDevCapacity);
        }
        __syncwarp();   // the keys and values have been read: the next row may write them
    }
}

// --------------------------------------------------- numeric: dense rows
// Work units: a dense row's P column chunks (of 2^cw_log2 <= W columns: W
// unless the plan needs more units than that leaves) are cut into G equal
// segments (G in {1, 2, 4, ..., kSegGrid}, chosen per flops class so that a
// unit carries a bounded share of flops); one warp owns a unit.  For each
// chunk of its segment the warp walks A(i,:) in order and, per entry, the part
// of B(k,:) inside the chunk, found from a cursor that the previous chunk left
// (the first cursor of a segment comes from segtab, the position of the first
// column >= the segment start in every B row).  Products go into a dense
// accumulator acc[W] with presence flags, in ascending k; the chunk is then
// emitted in column order.  Cursors live in a per-warp arena slot.


__host__ __device__ __forceinline__ long long seg_chunk(int g, int P) {
    return ((long long)g * P) / kSegGrid;
}

// Where a warp stands in B(k,:) while it sweeps the chunks of a row: the
// first unconsumed position, its column (INT_MAX once B(k,:) is used up) and
// its run length (entries from pos to the end of that column's chunk).
struct __align__(16) DenseCursor {
    long long pos;
    int col;
    int rl;
};

// Run tables of B, at the positions where a run (the entries of B(k,:) inside
// one column chunk, col >> cw_log2) starts: runlen[run_base + q] = its length,
// nextrun[run_base + q] = {length, first column} of the run after it ({0,
// INT_MAX} at the row's end), so a cursor advances with one load whose address
// it knows before the chunk's products are accumulated.  Other positions are not
// written: a cursor only ever stands at the start of a run.

// A run, as the entries before it need it: its chunk (-1: none, the row's end),
// its first column, where it ends, and the run after it.  Places count from the
// row's start.
struct RunAhead {
    int chunk, col, end;
    int2 next;
};

// The end of the run that place q of the row is in, by the whole warp.
template <class IT>
__device__ __forceinline__ int run_end(const IT* __restrict__ ci, int q, int len, int cw_log2) {
    const int ch = (int)(ci[q] >> cw_log2);
    int lo = q + 1, hi = len;   // the end is in [lo, hi]
    while (hi - lo > 32) {
        const int step = (hi - lo + 31) / 32;
        const int p = lo + (lane_id() + 1) * step - 1;
        const unsigned in = __ballot_sync(kFull, p < hi && (int)(ci[min(p, hi - 1)] >> cw_log2) == ch);
        const int k = __popc(in);
        hi = min(hi, lo + (k + 1) * step - 1);
        lo += k * step;
    }
    const int p = lo + lane_id();
    return lo + __popc(__ballot_sync(kFull, p < hi && (int)(ci[min(p, len - 1)] >> cw_log2) == ch));
}

// Places [a, b) of a row of `len` entries (ci, rl and nr start at the row), by a
// warp, from the end backwards: 128 entries per step, all loaded at once, and
// what a window's last run needs to know of the entries after it is carried from
// lane 0 of the window before.  Every column is read once and both tables are
// written from registers.
template <class IT>
__device__ __forceinline__ void run_tables_range(const IT* __restrict__ ci, int a, int b, int len,
                                                 int cw_log2, int32_t* __restrict__ rl,
                                                 int2* __restrict__ nr) {
    const int lane = lane_id();
    RunAhead ahead{-1, 0x7fffffff, len, make_int2(0, 0x7fffffff)};
    if (b < len) {
        ahead.col = (int)ci[b];
        ahead.chunk = ahead.col >> cw_log2;
        ahead.end = run_end(ci, b, len, cw_log2);
        if (ahead.end < len)
            ahead.next = make_int2(run_end(ci, ahead.end, len, cw_log2) - ahead.end,
                                   (int)ci[ahead.end]);
    }
    for (int hi = b; hi > a; hi -= 128) {
        // windows [hi - 32 u - 32, hi - 32 u) of lanes; places below a have no entry
        int col[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int q = hi - 32 * u - 32 + lane;
            col[u] = q >= a ? (int)ci[q] : -1;
        }
        const int first = hi - 128 > 0 ? (int)ci[hi - 129] : -1;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int lo = hi - 32 * u - 32;
            const int q = lo + lane;
            const int ch = col[u] >> cw_log2;
            int before = __shfl_up_sync(kFull, ch, 1);
            const int left = u < 3 ? __shfl_sync(kFull, col[u < 3 ? u + 1 : 3], 31) : first;
            if (lane == 0) before = left >> cw_log2;
            if (q == a) before = a > 0 ? (int)(ci[a - 1] >> cw_log2) : -1;
            const bool start = q >= a && before != ch;
            const unsigned later = __ballot_sync(kFull, start) & ~lanemask_le();
            const int t = __ffs(later) - 1;   // the next start in the window, if any
            int end = lo + t;
            if (later == 0u) end = ahead.chunk == ch ? ahead.end : lo + 32;
            int2 next;
            next.x = __shfl_sync(kFull, end - q, t & 31);
            next.y = __shfl_sync(kFull, col[u], t & 31);
            if (later == 0u) {
                if (ahead.chunk == ch) next = ahead.next;
                else next = make_int2(ahead.end - end, ahead.col);
            }
            if (start) {
                rl[q] = end - q;
                nr[q] = next;
            }
            if (lo <= a) break;
            ahead.chunk = __shfl_sync(kFull, ch, 0);
            ahead.col = __shfl_sync(kFull, col[u], 0);
            ahead.end = __shfl_sync(kFull, end, 0);
            ahead.next.x = __shfl_sync(kFull, next.x, 0);
            ahead.next.y = __shfl_sync(kFull, next.y, 0);
        }
    }
}

// A whole row, by a warp.  Rows of at most 32 entries are one window and need no
// carry.
template <class IT>
__device__ __forceinline__ void run_tables_row(const IT* __restrict__ ci, int len, int cw_log2,
                                               int32_t* __restrict__ rl, int2* __restrict__ nr) {
    if (len > 32) {
        run_tables_range<IT>(ci, 0, len, len, cw_log2, rl, nr);
        return;
    }
    const int q = lane_id();
    const int col = q < len ? (int)ci[q] : 0x7fffffff;
    const int before = __shfl_up_sync(kFull, col, 1);
    const bool start = q < len && (q == 0 || before >> cw_log2 != col >> cw_log2);
    const unsigned later = __ballot_sync(kFull, start) & ~lanemask_le();
    const int next = later ? __ffs(later) - 1 : len;
    const int next_len = __shfl_sync(kFull, next - q, next & 31);
    const int next_col = __shfl_sync(kFull, col, next & 31);
    if (start) {
        rl[q] = next - q;
        nr[q] = later ? make_int2(next_len, next_col) : make_int2(0, 0x7fffffff);
    }
}

template <class IT>
struct BRow {
    const IT* ci;
    long long s0, s1, run_base;
};

template <class IT>
__device__ __forceinline__ BRow<IT> b_row(const ProdDesc* __restrict__ D,
                                          const long long* __restrict__ bb, int nprod,
                                          long long kb) {
    const ProdDesc& d = D[nprod > 1 ? find_prod(bb, nprod, kb) : 0];
    const long long k = kb - d.brow_base;
    return BRow<IT>{(const IT*)d.ciB, d.rpB[k], d.rpB[k + 1], d.run_base};
}

// A warp per B row (inside the persistent chain).
template <class IT>
__device__ __forceinline__ void runlen_kernel_body(long long LB, const ProdDesc* __restrict__ D,
                              const long long* __restrict__ bb, int nprod, int cw_log2,
                              int32_t* __restrict__ runlen, int2* __restrict__ nextrun,
                              const DevCounters* cnt,
        const long long vbid, const long long vnb) {
    if (cnt->class_off[kNumClasses] == cnt->class_off[kClassDense0]) return;  // no dense rows
    const long long warp = ((long long)vbid * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)vnb * blockDim.x) >> 5;
    for (long long kb = warp; kb < LB; kb += nwarps) {
        const BRow<IT> r = b_row<IT>(D, bb, nprod, kb);
        run_tables_row<IT>(r.ci + r.s0, (int)(r.s1 - r.s0), cw_log2, runlen + r.run_base + r.s0,
                           nextrun + r.run_base + r.s0);
    }
}

// A warp per B row; eight, each a part of it, for a row of more than kRunLong.
// What bounds it: instructions and the stores (12 bytes per run).  Two passes
// per row, windows of 32 loaded one after another and a block for rows of more
// than 512 entries took, in us: R-MAT, 65536 vertices 83, now 35; scale 18 218
// and 123; the 0.75 G entries of a Markov step on 2^20 vertices, whose rows of
// 711 entries have runs of one or two, 10670 and 3610.  The limit, before the
// register cap: 1024 30, 119 and 4750; 2048 41, 142 and 4390; 4096 41, 143 and
// 4260.  The cap keeps six blocks resident (five without: 36, 129 and 3750; eight
// spill: 45, 141 and 3520).
constexpr int kRunLong = 2048;
template <class IT>
__global__ void __launch_bounds__(32 * kRowWarps, 6)
    runlen_kernel(long long LB, const ProdDesc* __restrict__ D,
                  const long long* __restrict__ bb, int nprod, int cw_log2,
                  int32_t* __restrict__ runlen, int2* __restrict__ nextrun,
                  const DevCounters* cnt) {
    if (cnt->class_off[kNumClasses] == cnt->class_off[kClassDense0]) return;  // no dense rows
    // as for_rows, but a row of a batch is looked up once
    __shared__ BRow<IT> longs[kRowWarps];
    const int w = threadIdx.x >> 5;
    for (long long tile = blockIdx.x; tile * kRowWarps < LB; tile += gridDim.x) {
        const long long kb = tile * kRowWarps + w;
        BRow<IT> r{nullptr, 0, 0, 0};
        if (kb < LB) r = b_row<IT>(D, bb, nprod, kb);
        const bool big = r.s1 - r.s0 > kRunLong;
        if (!big && r.s1 > r.s0)
            run_tables_row<IT>(r.ci + r.s0, (int)(r.s1 - r.s0), cw_log2, runlen + r.run_base + r.s0,
                               nextrun + r.run_base + r.s0);
        if (lane_id() == 0) longs[w] = big ? r : BRow<IT>{nullptr, 0, 0, 0};
        if (__syncthreads_or(big))
            for (int t = 0; t < kRowWarps; ++t) {
                const BRow<IT> x = longs[t];
                const int len = (int)(x.s1 - x.s0);
                const int per = ((len + kRowWarps - 1) / kRowWarps + 127) & ~127;
                const int from = min(len, per * w), to = min(len, from + per);
                if (from < to)
                    run_tables_range<IT>(x.ci + x.s0, from, to, len, cw_log2,
                                         runlen + x.run_base + x.s0, nextrun + x.run_base + x.s0);
            }
        __syncthreads();   // the list has been read
    }
}

// segtab[seg_base + k * (kSegGrid+1) + g] = first position p in B(k,:) with
// col >= seg_chunk(g, P) << cw_log2, relative to rowptr[k].
template <class IT>
__device__ __forceinline__ void segtab_kernel_body(long long LB, const ProdDesc* __restrict__ D,
                              const long long* __restrict__ bb, int nprod, int cw_log2,
                              int32_t* __restrict__ segtab, const DevCounters* cnt,
        const long long vbid, const long long vnb) {
    if (cnt->class_off[kNumClasses] == cnt->class_off[kClassDense0]) return;  // no dense rows
    const long long total = LB * (kSegGrid + 1);
    for (long long t = (long long)vbid * blockDim.x + threadIdx.x; t < total;
         t += (long long)vnb * blockDim.x) {
        const long long kb = t / (kSegGrid + 1);
        const int g = (int)(t - kb * (kSegGrid + 1));
        const int pr = nprod > 1 ? find_prod(bb, nprod, kb) : 0;
        const ProdDesc& d = D[pr];
        const long long k = kb - d.brow_base;
        const IT* ciB = (const IT*)d.ciB;
        const long long key = seg_chunk(g, d.P) << cw_log2;
        long long lo = d.rpB[k], hi = d.rpB[k + 1];
        const long long base = lo;
        while (lo < hi) {
            long long mid = (lo + hi) >> 1;
            if ((long long)ciB[mid] < key) lo = mid + 1;
            else hi = mid;
        }
        segtab[d.seg_base + k * (kSegGrid + 1) + g] = (int32_t)(lo - base);
    }
}

template <class IT>
__global__ void segtab_kernel(long long LB, const ProdDesc* __restrict__ D,
                              const long long* __restrict__ bb, int nprod, int cw_log2,
                              int32_t* __restrict__ segtab, const DevCounters* cnt) {
    segtab_kernel_body<IT>(LB, D, bb, nprod, cw_log2, segtab, cnt, (long long)blockIdx.x,
        (long long)gridDim.x);
}

// Products of one batch of (up to 32) A entries inside the chunk starting at
// column c0: lane e holds entry e's run (here, its B position pos, length len
// and a = A(i,k)).  The runs are flattened into rounds of 32 products in
// ascending k, four rounds per step so that their loads overlap; a round's
// products are multiplied and added in k order (lanes of one round that hit
// the same slot add in lane order, i.e. in ascending k).
template <class IT, class V>
__device__ __forceinline__ void dense_batch(bool here, long long pos, int len, V a, long long c0,
                                            const IT* __restrict__ ciB, const V* __restrict__ vB,
                                            V* acc, unsigned* bm, DenseRun<V>* runs) {
    const unsigned hmask = __ballot_sync(kFull, here);
    const int mylen = here ? len : 0;
    const int incl = warp_incl_scan(mylen);
    const int excl = incl - mylen;
    const int total = __shfl_sync(kFull, incl, 31);
    // nonempty runs in k order: run e starts at flattened position excl_e, its
    // products are B[off_e + f] for f in the run
    if (here) {
        DenseRun<V> re;
        re.off = pos - excl;
        re.a = a;
        runs[__popc(hmask & lanemask_lt())] = re;
    }
    __syncwarp();
    // The run of lane x in the round starting at w0 is (runs started before
    // w0) + (runs starting in [w0, w0 + x]) - 1, from an OR of start bits.
    int started = 0;
    for (int f0 = 0; f0 < total; f0 += 128) {
        const int nsub = min(4, (total - f0 + 31) >> 5);
        long long jj[4];
        V bv[4];
        V av[4];
        bool vl[4];
        bool multi[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            vl[t] = false;
            multi[t] = false;
            jj[t] = c0;
            bv[t] = V{};
            av[t] = V{};
            if (t < nsub) {
                const int w0 = f0 + 32 * t;
                const unsigned sbit =
                    (here && excl >= w0 && excl < w0 + 32) ? (1u << (excl - w0)) : 0u;
                const unsigned M = __reduce_or_sync(kFull, sbit);
                const int e = started + __popc(M & lanemask_le()) - 1;
                started += __popc(M);
                multi[t] = (M & ~1u) != 0u;
                const int fi = w0 + lane_id();
                vl[t] = fi < total;
                if (vl[t]) {
                    const DenseRun<V> re = runs[e];
                    const long long q = re.off + fi;
                    jj[t] = (long long)ciB[q];
                    bv[t] = load_val(vB, q);
                    av[t] = re.a;
                }
            }
        }
        V v[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            v[t] = V{};
            if (t < nsub && vl[t]) v[t] = VOps<V>::mul(av[t], bv[t]);
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            if (t < nsub) {
                const int slot = (int)(jj[t] - c0);
                if (vl[t]) atomicOr(&bm[slot >> 5], 1u << (slot & 31));
                if (multi[t]) ordered_add(acc, slot, vl[t], v[t]);
                else plain_add(acc, slot, vl[t], v[t]);
            }
        }
    }
    __syncwarp();
}

// The register cap (three 8-warp or six 4-warp blocks per SM) keeps 24
// warps resident, which the shared-memory accumulators allow.
template <class IT, class V, int W, int WARPS>
__device__ __forceinline__ void numeric_dense_kernel_body(
    const ProdDesc* __restrict__ D, const long long* __restrict__ rb,
                         int nprod, const int32_t* __restrict__ rows, const DevCounters* cnt,
                         const int32_t* __restrict__ chunkcnt, const int32_t* __restrict__ segtab,
                         const int32_t* __restrict__ runlen, const int2* __restrict__ nextrun,
                         DenseCursor* __restrict__ arena, long long arena_stride,
                         const int64_t* __restrict__ rpC, long long cap, IT* __restrict__ ciC,
                         V* __restrict__ vC, long long max_dense_n, unsigned long long* work,
                         int* err, int64_t* __restrict__ rowend, int32_t* __restrict__ overflow,
                         unsigned* overflow_count, int64_t* __restrict__ unit_cnt,
        const int cw_log2, const long long vbid, const long long vnb) {
    constexpr bool HV = VOps<V>::has_val;
    constexpr int kNone = 0x7fffffff;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = lane_id();
    const int w = threadIdx.x >> 5;
    constexpr size_t vbytes = HV ? sizeof(V) * W : 0;
    unsigned char* base = smem_raw + (size_t)w * (vbytes + W / 8 + 32 * sizeof(DenseRun<V>));
    V* acc = reinterpret_cast<V*>(base);
    unsigned* bm = reinterpret_cast<unsigned*>(base + vbytes);
    DenseRun<V>* runs = reinterpret_cast<DenseRun<V>*>(base + vbytes + W / 8);
    DenseCursor* cursor = arena + ((long long)vbid * WARPS + w) * arena_stride;
    for (int s = lane; s < W; s += 32)
        if constexpr (HV) acc[s] = VOps<V>::init();
    for (int s = lane; s < W / 32; s += 32) bm[s] = 0u;
    __syncwarp();
    const unsigned long long* ub = cnt->unit_begin;
    const long long total_units = (long long)ub[kMaxDenseClasses];
    const int32_t* drow = rows + cnt->class_off[kClassDense0];
    while (true) {
        long long u = 0;
        if (lane == 0) u = (long long)atomicAdd(work, 1ull);
        u = __shfl_sync(kFull, u, 0);
        if (u >= total_units) break;
        int b = 0;
        while (b + 1 < kMaxDenseClasses && (long long)ub[b + 1] <= u) ++b;
        const int G = dense_class_segments(b, cnt->seg_log2);
        const long long local = u - (long long)ub[b];
        const long long rr = (long long)(cnt->class_off[kClassDense0 + b] -
                                         cnt->class_off[kClassDense0]) + local / G;
        const int seg = (int)(local % G);
        const long long r = drow[rr];
        const RowCtx<IT, V> cx = row_ctx<IT, V>(D, rb, nprod, r);
        const int P = cx.P;
        const long long n = cx.n;
        if (n > max_dense_n) continue;
        const int g0 = seg * (kSegGrid / G);
        const int cs = (int)seg_chunk(g0, P);
        const int ce = (int)seg_chunk(g0 + kSegGrid / G, P);
        if (cs >= ce) continue;
        const long long a0 = cx.a0, a1 = cx.a1;
        if (a1 - a0 > arena_stride) {
            if (lane == 0) atomicExch(err, (int)kDevArena);
            continue;
        }
        const IT* ciA = cx.ciA;
        const V* vA = cx.vA;
        const int64_t* rpB = cx.rpB;
        const IT* ciB = cx.ciB;
        const V* vB = cx.vB;
        const int32_t* ccnt = chunkcnt + cx.chunk_base + cx.i * P;
        const int32_t* stab = segtab + cx.seg_base;
        const int32_t* rlen = runlen + cx.run_base;
        const int2* nrun = nextrun + cx.run_base;
        // Slot mode (learned sizing, no symbolic pass): the row's predicted
        // slot [rpC[r], rpC[r+1]) is split over its segments in proportion
        // to their chunks; a segment that outgrows its share lists the row
        // for an exact re-run.  Otherwise the chunk counts of the symbolic
        // pass give the segment's exact place in C.
        const bool slot_mode = rowend != nullptr;
        long long out, out_end;
        if (slot_mode) {
            const long long span = rpC[r + 1] - rpC[r];
            out = rpC[r] + span * cs / P;
            out_end = rpC[r] + span * ce / P;
        } else {
            long long before = 0;
            for (int c = lane; c < cs; c += 32) before += ccnt[c];
            before = warp_sum(before);
            out = rpC[r] + before;
            long long seg_total = 0;
            for (int c = cs + lane; c < ce; c += 32) seg_total += ccnt[c];
            seg_total = warp_sum(seg_total);
            if (seg_total == 0) continue;
            out_end = out + seg_total;
            if (out_end > cap) {
                if (lane == 0) atomicExch(err, (int)kDevCapacity);
                continue;
            }
        }
        const long long out_begin = out;
        // cursors at the segment start; the smallest column over all cursors
        // names the next chunk with any product, so chunks without products
        // are jumped over
        int min_next = kNone;
        for (long long p = a0 + lane; p < a1; p += 32) {
            const long long k = (long long)ciA[p];
            const long long s1 = rpB[k + 1];
            const long long c0p = g0 == 0 ? rpB[k] : rpB[k] + stab[k * (kSegGrid + 1) + g0];
            DenseCursor nc;
            nc.pos = c0p;
            nc.col = c0p < s1 ? (int)ciB[c0p] : kNone;
            nc.rl = c0p < s1 ? rlen[c0p] : 0;
            cursor[p - a0] = nc;
            min_next = min(min_next, nc.col);
        }
        min_next = warp_min(min_next);
        __syncwarp();
        for (int c = max(cs, min_next >> cw_log2); c < ce;) {
            const long long c0 = (long long)c << cw_log2;
            const long long c1 = min(c0 + (1LL << cw_log2), n);
            int cnext = kNone;  // smallest column after this chunk
            // batches of 32 entries: cursors and A values are loaded together
            // (neither address depends on the other); a cursor's next run is
            // loaded before the batch is accumulated and used after it
            for (long long bb = a0; bb < a1; bb += 32) {
                const long long p = bb + lane;
                DenseCursor cur{0, kNone, 0};
                V a = VOps<V>::init();
                if (p < a1) {
                    cur = cursor[p - a0];
                    a = load_val(vA, p);
                }
                const bool here = p < a1 && (long long)cur.col < c1;
                int2 nx = make_int2(0, kNone);
                if (here) nx = nrun[cur.pos];
                if (__any_sync(kFull, here))
                    dense_batch<IT, V>(here, cur.pos, cur.rl, a, c0, ciB, vB, acc, bm, runs);
                if (here) {
                    DenseCursor nc;
                    nc.pos = cur.pos + cur.rl;
                    nc.col = nx.y;
                    nc.rl = nx.x;
                    cursor[p - a0] = nc;
                    cnext = min(cnext, nc.col);
                } else {
                    cnext = min(cnext, cur.col);
                }
            }
            // emit the chunk in column order: lane t owns bitmap word t (32
            // columns), a warp scan of the popcounts gives each lane its output
            // run; words and values are reset on the way
            const int nwords = 1 << (cw_log2 - 5);
            for (int t0 = 0; t0 < nwords; t0 += 32) {
                const int wi0 = t0 + lane;
                unsigned word = wi0 < nwords ? bm[wi0] : 0u;
                const int pc = __popc(word);
                const int pincl = warp_incl_scan(pc);
                long long pos = out + (pincl - pc);
                while (word) {
                    const int bit = __ffs(word) - 1;
                    word &= word - 1;
                    const int s = wi0 * 32 + bit;
                    if (pos < out_end) {
                        ciC[pos] = (IT)(c0 + s);
                        if constexpr (HV) vC[pos] = acc[s];
                    }
                    if constexpr (HV) acc[s] = VOps<V>::init();
                    ++pos;
                }
                if (wi0 < nwords) bm[wi0] = 0u;
                out += __shfl_sync(kFull, pincl, 31);
            }
            __syncwarp();
            const int jump = warp_min(cnext) >> cw_log2;
            c = max(c + 1, jump);
        }
        if (lane == 0) {
            if (!slot_mode) {
                if (out != out_end) atomicExch(err, (int)kDevCountMismatch);
            } else if (out > out_end) {
                if (atomicCAS((unsigned long long*)&rowend[r], 0ull, ~0ull) == 0ull)
                    overflow[atomicAdd(overflow_count, 1u)] = (int32_t)r;
            } else {
                unit_cnt[u] = out - out_begin;
            }
        }
    }
}

template <class IT, class V, int W, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, 24 / WARPS)
    numeric_dense_kernel(const ProdDesc* __restrict__ D, const long long* __restrict__ rb,
                         int nprod, const int32_t* __restrict__ rows, const DevCounters* cnt,
                         const int32_t* __restrict__ chunkcnt, const int32_t* __restrict__ segtab,
                         const int32_t* __restrict__ runlen, const int2* __restrict__ nextrun,
                         DenseCursor* __restrict__ arena, long long arena_stride,
                         const int64_t* __restrict__ rpC, long long cap, IT* __restrict__ ciC,
                         V* __restrict__ vC, long long max_dense_n, unsigned long long* work,
                         int* err, int64_t* __restrict__ rowend, int32_t* __restrict__ overflow,
                         unsigned* overflow_count, int64_t* __restrict__ unit_cnt, int cw_log2) {
    numeric_dense_kernel_body<IT, V, W, WARPS>(D, rb, nprod, rows, cnt, chunkcnt, segtab, runlen,
        nextrun, arena, arena_stride, rpC, cap, ciC, vC, max_dense_n, work, err, rowend,
        overflow, overflow_count, unit_cnt, cw_log2, (long long)blockIdx.x, (long long)gridDim.x);
}

// Learned sizing: close the gaps a slot-mode dense row leaves between its
// segments (each segment moves left to follow the previous one) and set
// rowend.  One warp per dense row; rows listed for a re-run are skipped.
template <class IT, class V>
__global__ void dense_slot_pack_kernel(const ProdDesc* __restrict__ D,
                                       const long long* __restrict__ rb, int nprod,
                                       const int32_t* __restrict__ rows,
                                       const DevCounters* __restrict__ cnt,
                                       const int64_t* __restrict__ rpC,
                                       const int64_t* __restrict__ unit_cnt,
                                       int64_t* __restrict__ rowend, IT* __restrict__ ciC,
                                       V* __restrict__ vC) {
    constexpr bool HV = VOps<V>::has_val;
    const int lane = lane_id();
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    const long long d0 = (long long)cnt->class_off[kClassDense0];
    const long long nd = (long long)cnt->class_off[kNumClasses] - d0;
    const unsigned long long* ub = cnt->unit_begin;
    for (long long rr = warp; rr < nd; rr += nwarps) {
        int b = 0;
        while (b + 1 < kMaxDenseClasses &&
               (long long)cnt->class_off[kClassDense0 + b + 1] - d0 <= rr)
            ++b;
        const int G = dense_class_segments(b, cnt->seg_log2);
        const long long local = rr - ((long long)cnt->class_off[kClassDense0 + b] - d0);
        const long long u0 = (long long)ub[b] + local * G;
        const long long r = rows[d0 + rr];
        if (rowend[r] != 0) continue;  // listed for a re-run
        const int P = D[nprod > 1 ? find_prod(rb, nprod, r) : 0].P;
        const long long start = rpC[r];
        const long long span = rpC[r + 1] - start;
        long long dst = start;
        for (int g = 0; g < G; ++g) {
            const int g0 = g * (kSegGrid / G);
            const long long src = start + span * seg_chunk(g0, P) / P;
            const long long len = unit_cnt[u0 + g];
            if (src != dst) {
                // dst < src: a forward copy in steps of 128 entries (all of a
                // step read before any is written) never overwrites an entry
                // before it is read; four loads per lane are in flight
                for (long long q = 0; q < len; q += 128) {
                    IT cv[4];
                    V vv[4];
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        const long long x = q + 32 * t + lane;
                        cv[t] = IT{};
                        vv[t] = V{};
                        if (x < len) {
                            cv[t] = ciC[src + x];
                            if constexpr (HV) vv[t] = vC[src + x];
                        }
                    }
                    __syncwarp();
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        const long long x = q + 32 * t + lane;
                        if (x < len) {
                            ciC[dst + x] = cv[t];
                            if constexpr (HV) vC[dst + x] = vv[t];
                        }
                    }
                    __syncwarp();
                }
            }
            dst += len;
        }
        if (lane == 0) rowend[r] = dst;
    }
}

// ------------------------------------------------------------ k-slices
// bounds[s*m + i] = first position in A(i,:) with column >= floor(s*l/c).
template <class IT>
__global__ void kslice_bounds_kernel(long long m, long long l, int c,
                                     const int64_t* __restrict__ rp, const IT* __restrict__ ci,
                                     int64_t* __restrict__ bounds) {
    const long long total = m * (long long)(c + 1);
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const long long s = t / m, i = t - s * m;
        const long long key = (s * l) / c;
        long long lo = rp[i], hi = rp[i + 1];
        while (lo < hi) {
            long long mid = (lo + hi) >> 1;
            if ((long long)ci[mid] < key) lo = mid + 1;
            else hi = mid;
        }
        bounds[t] = lo;
    }
}

}  // namespace sg
