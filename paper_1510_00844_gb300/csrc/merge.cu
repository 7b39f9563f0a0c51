// Sum of c partial products C = sum_s C_s, entries with equal (i, j) added in
// ascending s: the result of the paper's multiway merge with duplicate
// reduction (Sec. 4.3), used for the LocalMerge of the k-slice partials
// (Alg. 2).  The paper merges sorted triple lists with a heap of size c; here
// one warp owns a row (or a column segment of a long one) and takes it in
// chunks of at most S entries over all lists: each list offers a share of the
// next S entries in proportion to what it has left, and the chunk ends at the
// smallest column that a list could not offer.  The chunk's columns set bits
// in a column map; the bits before a column are its place among the chunk's
// outputs, so the accumulator holds outputs and not columns.  The lists' values
// are then added in order s = 0..c-1 (a list has distinct columns, so 32 of
// its entries never repeat a place) and the chunk is written, all lanes side
// by side.
//
// Rows of more than kMergeLong entries are listed and cut into kMergeSegs
// column segments: a power-law graph's longest row holds more entries than a
// warp should add while the others have finished.
//
// What bounds it: the count, instructions (issue 82 % active); the numeric pass,
// instructions and the latency of a chunk's few dependent steps (columns, map,
// values) at 20 warps per SM (issue 53 %, DRAM 21 %).  The sweep of 1024-column chunks that
// this replaces met few entries per chunk on rows of ordinary length and left
// the longest rows to single warps.  Before and now: four lists of 100003-vertex
// R-MAT graphs (3.3 GB read and written) 5.70 and 2.80 ms; the four partial
// products of a 65536-vertex graph squared (11 GB) 8.9 and 7.1 ms; nine
// partial products 40.6 and 13.0 ms.
#include <type_traits>

#include "plan.h"

namespace sg {

constexpr int kMaxMergeParts = 32;
constexpr int kMergeWarps = 4;
// Columns a chunk may span, and the most entries it takes: the numeric pass
// holds an accumulator and two 16-bit columns per entry, the count only bits.
// More of either costs warps: twice the span 2.8 and 7.9 ms, twice the span
// and the entries 3.2 and 8.8 ms for the first two figures above.
constexpr int kMergeSpan = 16384;
constexpr int kMergeS = 512;
constexpr int kMergeCountS = 2048;

template <class IT, class V>
struct MergeParts {
    const int64_t* rp[kMaxMergeParts];
    const int64_t* re[kMaxMergeParts];
    const IT* col[kMaxMergeParts];
    const V* val[kMaxMergeParts];
    long long len[kMaxMergeParts];  // length of col/val of part s
};

// (+, x) stores the first list's values instead of adding them to the identity.
template <class V>
constexpr bool kStoreFirst = std::is_same<V, double>::value || std::is_same<V, float>::value ||
                             std::is_same<V, int64_t>::value;

// Shared memory of a warp: accumulators, the column map (bits, and for the
// numeric pass the outputs before each word), the chunk's columns in list
// order and in output order (offsets from its first column).
template <class V, bool NUMERIC>
struct MergeWarp {
    static constexpr int kWords = kMergeSpan / 32;
    static constexpr int kS = NUMERIC ? kMergeS : kMergeCountS;
    static constexpr size_t kBitsAt = NUMERIC && VOps<V>::has_val ? sizeof(V) * kS : 0;
    static constexpr size_t kBeforeAt = kBitsAt + sizeof(unsigned) * kWords;
    static constexpr size_t kListAt = kBeforeAt + (NUMERIC ? sizeof(unsigned short) * kWords : 0);
    static constexpr size_t kOutAt = kListAt + (NUMERIC ? sizeof(unsigned short) * kS : 0);
    static constexpr size_t kBytes = kOutAt + (NUMERIC ? sizeof(unsigned short) * kS : 0);
};

// One row's (or segment's) merge by a warp: lane s holds list s's range
// [cur, end).  Returns the number of outputs; writes them from `out` on
// (numeric; never at or past out_end).  Rows must ascend; a row that does not
// gives a wrong sum, or -1 where a chunk could take nothing.  Whatever the columns
// are, every chunk takes an entry, only offsets below the span reach the map and
// the list, and a value's place is below the chunk's outputs.  (Testing every 32
// entries for the order cost 11 % of a merge of four 100003-vertex graphs,
// testing for columns below c0 17 %; these bounds cost nothing.)
template <class IT, class V, bool NUMERIC>
__device__ __forceinline__ long long merge_range(int c, const MergeParts<IT, V>& parts,
                                                 long long cur, long long end, long long out,
                                                 long long out_end, IT* __restrict__ ciC,
                                                 V* __restrict__ vC, unsigned char* smem) {
    using L = MergeWarp<V, NUMERIC>;
    constexpr bool HV = NUMERIC && VOps<V>::has_val;
    constexpr long long kFar = 0x7fffffffffffffffLL;
    V* acc = reinterpret_cast<V*>(smem);
    unsigned* bits = reinterpret_cast<unsigned*>(smem + L::kBitsAt);
    unsigned short* before = reinterpret_cast<unsigned short*>(smem + L::kBeforeAt);
    unsigned short* list = reinterpret_cast<unsigned short*>(smem + L::kListAt);
    unsigned short* outs = reinterpret_cast<unsigned short*>(smem + L::kOutAt);
    const int lane = lane_id();
    using U = typename std::make_unsigned<IT>::type;
    const IT* mycol = lane < c ? parts.col[lane] : nullptr;
    long long count = 0;
    // each list's share of the next chunk, its first column and the column
    // after its share: loaded as soon as the chunk before has taken its part
    long long total = 0, share = 0, head = kFar, next = kFar;
    auto offer = [&]() {
        const long long left = max(0LL, end - cur);
        total = warp_sum(left);
        share = left;
        if (total > L::kS) share = min(left, (long long)(L::kS - 8 * c) * left / total + 8);
        head = left > 0 ? (long long)mycol[cur] : kFar;
        next = share < left ? (long long)mycol[cur + share] : kFar;
    };
    offer();
    while (total > 0) {
        const long long c0 = warp_min(head);
        const long long c1 = min(warp_min(next), c0 + kMergeSpan);
        if (c1 <= c0) return -1;
        const U width = (U)(c1 - c0);
        // columns: bits of the map, offsets in list order; four lists' loads
        // are in flight together
        int mine = 0;     // entries of list `lane` in the chunk
        int base = 0;
        int top = 0;      // one past the largest offset
        for (int s0 = 0; s0 < c; s0 += 4) {
            const IT* col[4];
            int lim[4];
            IT j[4][4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int s = min(s0 + u, c - 1);
                lim[u] = s0 + u < c ? __shfl_sync(kFull, (int)share, s) : 0;
                col[u] = parts.col[s] + __shfl_sync(kFull, cur, s);
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    j[u][t] = 32 * t + lane < lim[u] ? col[u][32 * t + lane] : IT(0);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                int n = 0;
                for (int x0 = 0; x0 < lim[u]; x0 += 128) {
                    if (x0 > 0) {
#pragma unroll
                        for (int t = 0; t < 4; ++t)
                            j[u][t] = x0 + 32 * t + lane < lim[u] ? col[u][x0 + 32 * t + lane] : IT(0);
                    }
                    int got = 0;
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        // a column below c0 wraps around to far above the width
                        const U off = (U)j[u][t] - (U)c0;
                        const bool in = x0 + 32 * t + lane < lim[u] && off < width;
                        if (in) {
                            const int d = (int)off;
                            atomicOr(&bits[d >> 5], 1u << (d & 31));
                            if constexpr (HV) list[base + x0 + 32 * t + lane] = (unsigned short)d;
                            top = max(top, d + 1);
                        }
                        got += __popc(__ballot_sync(kFull, in));
                    }
                    n += got;
                    if (got < 128) break;
                }
                mine = lane == s0 + u ? n : mine;
                base += n;
            }
        }
        const long long from = cur;   // where the chunk's part of list `lane` begins
        cur += mine;
        offer();
        const int nwords = ((int)__reduce_max_sync(kFull, (unsigned)top) + 31) >> 5;
        __syncwarp();
        if constexpr (!NUMERIC) {
            for (int t = lane; t < nwords; t += 32) {
                count += __popc(bits[t]);
                bits[t] = 0u;
            }
            __syncwarp();
            continue;
        }
        // outputs before each word; without values the columns are written here
        int n_out = 0;
        for (int w0 = 0; w0 < nwords; w0 += 128) {
            uint4 x = *reinterpret_cast<const uint4*>(bits + w0 + 4 * lane);
            const int p0 = __popc(x.x), p1 = p0 + __popc(x.y), p2 = p1 + __popc(x.z),
                      p3 = p2 + __popc(x.w);
            const int incl = warp_incl_scan(p3);
            const int b = n_out + incl - p3;
            ushort4 y;
            y.x = (unsigned short)b;
            y.y = (unsigned short)(b + p0);
            y.z = (unsigned short)(b + p1);
            y.w = (unsigned short)(b + p2);
            *reinterpret_cast<ushort4*>(before + w0 + 4 * lane) = y;
            n_out += __shfl_sync(kFull, incl, 31);
        }
        __syncwarp();
        if constexpr (HV) {
            base = 0;
            for (int s0 = 0; s0 < c; s0 += 4) {
                const V* val[4];
                int n[4];
                V v[4][4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int s = min(s0 + u, c - 1);
                    n[u] = s0 + u < c ? __shfl_sync(kFull, mine, s) : 0;
                    val[u] = parts.val[s] + __shfl_sync(kFull, from, s);
#pragma unroll
                    for (int t = 0; t < 4; ++t)
                        if (32 * t + lane < n[u]) v[u][t] = val[u][32 * t + lane];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    for (int x0 = 0; x0 < n[u]; x0 += 128) {
                        if (x0 > 0) {
#pragma unroll
                            for (int t = 0; t < 4; ++t)
                                if (x0 + 32 * t + lane < n[u]) v[u][t] = val[u][x0 + 32 * t + lane];
                        }
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            const int x = x0 + 32 * t + lane;
                            if (x < n[u]) {
                                const int d = list[base + x];
                                const int slot =
                                    min((int)before[d >> 5] +
                                            __popc(bits[d >> 5] & ~(0xffffffffu << (d & 31))),
                                        n_out - 1);
                                if (kStoreFirst<V> && s0 + u == 0) acc[slot] = v[u][t];
                                else acc[slot] = VOps<V>::add(acc[slot], v[u][t]);
                                outs[slot] = (unsigned short)d;
                            }
                        }
                    }
                    base += n[u];
                    __syncwarp();
                }
            }
        } else {
            // the places of the columns from the bits alone
            for (int t = lane; t < nwords; t += 32) {
                int p = before[t];
                for (unsigned word = bits[t]; word; word &= word - 1u)
                    outs[p++] = (unsigned short)(32 * t + __ffs(word) - 1);
            }
            __syncwarp();
        }
        for (int t = lane; t < n_out; t += 32) {
            const long long pos = out + count + t;
            if (pos < out_end) {
                ciC[pos] = (IT)(c0 + outs[t]);
                if constexpr (HV) vC[pos] = acc[t];
            }
            if constexpr (HV) acc[t] = VOps<V>::init();
        }
        for (int t = lane; t < nwords; t += 32) bits[t] = 0u;
        __syncwarp();
        count += n_out;
    }
    if constexpr (!NUMERIC) count = warp_sum(count);
    return count;
}

template <class IT, class V, bool NUMERIC>
__device__ __forceinline__ unsigned char* merge_warp_memory(unsigned char* smem_raw) {
    using L = MergeWarp<V, NUMERIC>;
    unsigned char* smem = smem_raw + (size_t)(threadIdx.x >> 5) * L::kBytes;
    if constexpr (NUMERIC && VOps<V>::has_val) {
        V* acc = reinterpret_cast<V*>(smem);
        for (int t = lane_id(); t < L::kS; t += 32) acc[t] = VOps<V>::init();
    }
    unsigned* bits = reinterpret_cast<unsigned*>(smem + L::kBitsAt);
    for (int t = lane_id(); t < L::kWords; t += 32) bits[t] = 0u;
    if constexpr (NUMERIC) {
        // offsets and places that no chunk has written are in bounds too
        unsigned short* before = reinterpret_cast<unsigned short*>(smem + L::kBeforeAt);
        unsigned short* list = reinterpret_cast<unsigned short*>(smem + L::kListAt);
        for (int t = lane_id(); t < L::kWords; t += 32) before[t] = 0;
        for (int t = lane_id(); t < L::kS; t += 32) list[t] = 0;
    }
    __syncwarp();
    return smem;
}

// Rows, one at a time per warp from a counter (row sizes are heavy-tailed).
// Rows of more than kMergeLong entries are put on `longs` (if given) while it
// has room, and left to the segment kernels.
template <class IT, class V, bool NUMERIC>
__global__ void __launch_bounds__(kMergeWarps * 32)
    merge_rows_kernel(int c, MergeParts<IT, V> parts, long long m, int64_t* __restrict__ rowcnt,
                      const int64_t* __restrict__ rpC, IT* __restrict__ ciC, V* __restrict__ vC,
                      int* err, unsigned long long* work, MergeLong* longs) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char* smem = merge_warp_memory<IT, V, NUMERIC>(smem_raw);
    const int lane = lane_id();
    while (true) {
        long long i = 0;
        if (lane == 0) i = (long long)atomicAdd(work, 1ull);
        i = __shfl_sync(kFull, i, 0);
        if (i >= m) break;
        long long cur = 0, end = 0;
        if (lane < c) {
            cur = parts.rp[lane][i];
            end = parts.re[lane] ? parts.re[lane][i] : parts.rp[lane][i + 1];
        }
        if (longs && warp_sum(end - cur) > kMergeLong) {
            unsigned at = 0;
            if (lane == 0) at = atomicAdd(&longs->count, 1u);
            at = __shfl_sync(kFull, at, 0);
            if (at < kMergeLongRows) {
                if (lane == 0) {
                    longs->row[at] = i;
                    if constexpr (!NUMERIC) rowcnt[i] = 0;
                }
                continue;
            }
        }
        const long long out = NUMERIC ? rpC[i] : 0, out_end = NUMERIC ? rpC[i + 1] : 0;
        const long long got =
            merge_range<IT, V, NUMERIC>(c, parts, cur, end, out, out_end, ciC, vC, smem);
        if (lane == 0) {
            if (got < 0) atomicExch(err, (int)kDevBadIndex);
            if constexpr (!NUMERIC) rowcnt[i] = max(0LL, got);
            else if (got >= 0 && out + got != out_end) atomicExch(err, (int)kDevCountMismatch);
        }
    }
}

// The listed rows: a warp takes one column segment of one row.  NUMERIC:
// places follow from the counts of the row's earlier segments; else the
// segment's outputs are counted (and added to the row's count, if wanted).
template <class IT, class V, bool NUMERIC>
__global__ void __launch_bounds__(kMergeWarps * 32)
    merge_segments_kernel(int c, MergeParts<IT, V> parts, int64_t* __restrict__ rowcnt, const int64_t* __restrict__ rpC,
                          IT* __restrict__ ciC, V* __restrict__ vC, int* err,
                          unsigned long long* work, MergeLong* longs) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char* smem = merge_warp_memory<IT, V, NUMERIC>(smem_raw);
    const int lane = lane_id();
    const long long units = (long long)min(longs->count, (unsigned)kMergeLongRows) * kMergeSegs;
    while (true) {
        long long u = 0;
        if (lane == 0) u = (long long)atomicAdd(work, 1ull);
        u = __shfl_sync(kFull, u, 0);
        if (u >= units) break;
        const int g = (int)(u % kMergeSegs);
        const long long i = longs->row[u / kMergeSegs];
        long long cur = 0, end = 0, lo = 0x7fffffffffffffffLL, hi = 0;
        const IT* col = nullptr;
        if (lane < c) {
            col = parts.col[lane];
            cur = parts.rp[lane][i];
            end = parts.re[lane] ? parts.re[lane][i] : parts.rp[lane][i + 1];
            if (cur < end) {
                lo = (long long)col[cur];
                hi = (long long)col[end - 1] + 1;
            }
        }
        // the row's columns [lo, hi) cut into equal segments
        lo = warp_min(lo);
        hi = warp_max(hi);
        const long long per = (hi - lo) / kMergeSegs, rest = (hi - lo) % kMergeSegs;
        auto bound = [&](int t) { return lo + per * t + rest * t / kMergeSegs; };
        auto first_from = [&](long long p, long long e, long long key) {
            while (p < e) {
                const long long mid = (p + e) >> 1;
                if ((long long)col[mid] < key) p = mid + 1;
                else e = mid;
            }
            return p;
        };
        if (g > 0) cur = first_from(cur, end, bound(g));
        if (g + 1 < kMergeSegs) end = first_from(cur, end, bound(g + 1));
        __syncwarp();
        long long out = 0, out_end = 0;
        if constexpr (NUMERIC) {
            const long long k = lane < kMergeSegs ? longs->seg[u / kMergeSegs * kMergeSegs + lane] : 0;
            out = rpC[i] + warp_sum(lane < g ? k : 0);
            out_end = min(out + __shfl_sync(kFull, k, g), (long long)rpC[i + 1]);
        }
        const long long got =
            merge_range<IT, V, NUMERIC>(c, parts, cur, end, out, out_end, ciC, vC, smem);
        if (got < 0) {   // the row's columns do not ascend
            if (lane == 0) {
                atomicExch(err, (int)kDevBadIndex);
                if constexpr (!NUMERIC) longs->seg[u] = 0;
            }
            continue;
        }
        if (lane == 0) {
            if constexpr (NUMERIC) {
                if (out + got != out_end || (g + 1 == kMergeSegs && out_end != rpC[i + 1]))
                    atomicExch(err, (int)kDevCountMismatch);
            } else {
                longs->seg[u] = got;
                if (rowcnt) atomicAdd((unsigned long long*)&rowcnt[i], (unsigned long long)got);
            }
        }
    }
}

// ------------------------------------------------ staged numeric merge
// The numeric sum for c <= CM lists whose column and value arrays start on
// 16-byte boundaries, with every list's entries staged in shared memory by
// bulk asynchronous copies (cp.async.bulk, the TMA's one-dimensional form):
// each warp keeps two buffers of WIN entries per list; while the warp
// accumulates from one, the next window of that list is in flight into the
// other, so each list has up to 2 x WIN entries in flight with no registers
// held.  A buffer's copy signals an mbarrier (transaction count = its
// bytes); the warp waits on it with a bound (a wait that exceeds the bound
// records kDevWaitTimeout, lets the copies it issued land, and ends the
// warp's work).  Windows start at multiples of four entries (16 bytes of
// int32 columns, 32 of float64 values); the last entries of an array that a
// 16-byte copy cannot reach are loaded by the lanes.  Entries are
// then consumed in column order, chunk by chunk of W columns.
__device__ __forceinline__ unsigned smem_u32(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(unsigned long long* bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
}

// One arrival that also expects `bytes` of asynchronous copies.
__device__ __forceinline__ void mbar_arrive_tx(unsigned long long* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void bulk_to_shared(void* dst, const void* src, unsigned bytes,
                                               unsigned long long* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ bool mbar_test(unsigned long long* bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

constexpr unsigned long long kMergeWaitNs = 2000000000ull;   // 2 s

// Bounded wait for the phase of `bar` with the given parity.
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity) {
    if (mbar_test(bar, parity)) return true;
    unsigned long long t0;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    while (true) {
        if (mbar_test(bar, parity)) return true;
        unsigned long long t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t - t0 > kMergeWaitNs) return false;
    }
}

template <class IT, class V, int W, int WARPS, int CM, int WIN>
struct MergeStage {
    static constexpr bool HV = VOps<V>::has_val;
    static constexpr size_t vbytes = HV ? sizeof(V) * W : 0;
    static constexpr size_t bufbytes = (size_t)WIN * (sizeof(IT) + (HV ? sizeof(V) : 0));
    // per warp: accumulator, bitmap, barriers, then 2 buffers per list (16-byte aligned)
    static constexpr size_t head = (vbytes + W / 8 + 16 * CM + 15) / 16 * 16;
    static constexpr size_t warp_bytes = head + 2 * CM * bufbytes;
};

template <class IT, class V, int W, int WARPS, int CM, int WIN>
__global__ void __launch_bounds__(WARPS * 32)
    merge_stage_kernel(int c, MergeParts<IT, V> parts, long long m, long long n,
                       const int64_t* __restrict__ rpC, IT* __restrict__ ciC, V* __restrict__ vC,
                       int* err, unsigned long long* work) {
    using L = MergeStage<IT, V, W, WARPS, CM, WIN>;
    constexpr bool HV = L::HV;
    constexpr int NWORDS = W / 32;
    static_assert(WIN % 32 == 0, "windows hold whole rounds of 32 entries");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = lane_id();
    const int w = threadIdx.x >> 5;
    unsigned char* base = smem_raw + (size_t)w * L::warp_bytes;
    V* acc = reinterpret_cast<V*>(base);
    unsigned* bm = reinterpret_cast<unsigned*>(base + L::vbytes);
    unsigned long long* bar = reinterpret_cast<unsigned long long*>(base + L::vbytes + W / 8);
    unsigned char* bufs = base + L::head;
    auto bcol = [&](int s, int b) {
        return reinterpret_cast<IT*>(bufs + (size_t)(2 * s + b) * L::bufbytes);
    };
    auto bval = [&](int s, int b) {
        return reinterpret_cast<V*>(bufs + (size_t)(2 * s + b) * L::bufbytes + WIN * sizeof(IT));
    };
    for (int t = lane; t < W; t += 32)
        if constexpr (HV) acc[t] = VOps<V>::init();
    for (int t = lane; t < NWORDS; t += 32) bm[t] = 0u;
    if (lane < 2 * CM) mbar_init(&bar[lane]);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    unsigned parity = 0u;   // bit 2s+b: parity of buffer b of list s's next phase
    unsigned pending = 0u;  // bit 2s+b: buffer b of list s has a copy in flight
    // lane 0 stages window [ws, ws + WIN) of list s (clipped to the row end
    // rounded up to four entries) into buffer b
    auto issue = [&](int s, int b, long long ws, long long e) {
        pending |= 1u << (2 * s + b);
        const long long len = parts.len[s];
        const long long we = min(ws + WIN, (e + 3) & ~3LL);
        const long long wc = max(ws, min(we, len & ~3LL));   // end of the 16-byte copies
        if (lane == 0) {
            const unsigned nb = (unsigned)(wc - ws);
            unsigned bytes = nb * (unsigned)sizeof(IT);
            if constexpr (HV) bytes += nb * (unsigned)sizeof(V);
            mbar_arrive_tx(&bar[2 * s + b], bytes);
            if (nb > 0) {
                bulk_to_shared(bcol(s, b), parts.col[s] + ws, nb * (unsigned)sizeof(IT),
                               &bar[2 * s + b]);
                if constexpr (HV)
                    bulk_to_shared(bval(s, b), parts.val[s] + ws, nb * (unsigned)sizeof(V),
                                   &bar[2 * s + b]);
            }
        }
        // the array's last entries past the copies, if the window reaches them
        const long long q = wc + lane;
        if (q < min(we, e) && q < len) {
            bcol(s, b)[q - ws] = parts.col[s][q];
            if constexpr (HV) bval(s, b)[q - ws] = parts.val[s][q];
        }
    };
    bool ok = true;
    while (ok) {
        long long i = 0;
        if (lane == 0) i = (long long)atomicAdd(work, 1ull);
        i = __shfl_sync(kFull, i, 0);
        if (i >= m) break;
        long long b_own = 0, e_own = 0;
        if (lane < c) {
            b_own = parts.rp[lane][i];
            e_own = parts.re[lane] ? parts.re[lane][i] : parts.rp[lane][i + 1];
        }
        long long pos[CM], end[CM], bst[CM];
        int cur[CM];
        // the previous row's reads of the buffers come before the new copies
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
#pragma unroll
        for (int s = 0; s < CM; ++s) {
            pos[s] = s < c ? __shfl_sync(kFull, b_own, s) : 0;
            end[s] = s < c ? __shfl_sync(kFull, e_own, s) : 0;
            bst[s] = pos[s] & ~3LL;
            cur[s] = 0;
            if (pos[s] < end[s]) {
                issue(s, 0, bst[s], end[s]);
                if (bst[s] + WIN < end[s]) issue(s, 1, bst[s] + WIN, end[s]);
            }
        }
        __syncwarp();
        // wait for a buffer's copy and take its phase
        auto take = [&](int s, int b) {
            const int t = 2 * s + b;
            if (!mbar_wait(&bar[t], (parity >> t) & 1u)) return false;
            parity ^= 1u << t;
            pending &= ~(1u << t);
            return true;
        };
#pragma unroll
        for (int s = 0; s < CM; ++s)
            if (ok && pos[s] < end[s]) ok = take(s, 0);
        if (!ok) break;
        long long out = rpC[i];
        const long long out_end = rpC[i + 1];
        while (ok) {
            long long nxt = n;
#pragma unroll
            for (int s = 0; s < CM; ++s)
                if (pos[s] < end[s]) nxt = min(nxt, (long long)bcol(s, cur[s])[pos[s] - bst[s]]);
            if (nxt >= n) break;
            const long long c0 = (nxt / W) * W;
            const long long c1 = min(c0 + (long long)W, n);
#pragma unroll
            for (int s = 0; s < CM; ++s) {
                while (ok && pos[s] < end[s]) {
                    const long long lim = min(bst[s] + WIN, end[s]);
                    const long long q = pos[s] + lane;
                    const IT* cb = bcol(s, cur[s]);
                    bool valid = q < lim;
                    long long col = 0;
                    if (valid) {
                        col = (long long)cb[q - bst[s]];
                        valid = col >= c0 && col < c1;
                    }
                    if (valid) {
                        const int slot = (int)(col - c0);
                        atomicOr(&bm[slot >> 5], 1u << (slot & 31));
                        if constexpr (HV) {
                            const V v = bval(s, cur[s])[q - bst[s]];
                            if (kStoreFirst<V> && s == 0) acc[slot] = v;
                            else acc[slot] = VOps<V>::add(acc[slot], v);
                        }
                    }
                    __syncwarp();
                    const int got = __popc(__ballot_sync(kFull, valid));
                    pos[s] += got;
                    if (pos[s] >= end[s]) break;          // the row's entries of list s are done
                    if (pos[s] < lim) {
                        if (got < 32) break;              // the chunk ends inside the buffer
                        continue;                         // a full round: the chunk may go on
                    }
                    // buffer used up (pos == bst + WIN < end): the other buffer holds
                    // the next window; this one is refilled with the window after it
                    const long long nw = bst[s] + 2 * WIN;
                    if (nw < end[s]) {
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        issue(s, cur[s], nw, end[s]);
                        __syncwarp();
                    }
                    cur[s] ^= 1;
                    bst[s] += WIN;
                    ok = take(s, cur[s]);
                }
            }
            if (!ok) break;
            // emit the chunk in column order, clearing it
            for (int t0 = 0; t0 < NWORDS; t0 += 32) {
                const int t = t0 + lane;
                unsigned word = t < NWORDS ? bm[t] : 0u;
                const int pc = __popc(word);
                const int incl = warp_incl_scan(pc);
                long long p = out + incl - pc;
                while (word) {
                    const int bit = __ffs(word) - 1;
                    word &= word - 1;
                    const int slot = t * 32 + bit;
                    if (p < out_end) {
                        ciC[p] = (IT)(c0 + slot);
                        if constexpr (HV) vC[p] = acc[slot];
                    }
                    if constexpr (HV) acc[slot] = VOps<V>::init();
                    ++p;
                }
                if (t < NWORDS) bm[t] = 0u;
                out += __shfl_sync(kFull, incl, 31);
            }
            __syncwarp();
        }
        if (ok && lane == 0 && out != out_end) atomicExch(err, (int)kDevCountMismatch);
    }
    if (!ok) {
        if (lane == 0) atomicExch(err, (int)kDevWaitTimeout);
        // let the copies this warp still has in flight land before it ends
        // (each wait bounded again)
        for (int t = 0; t < 2 * CM; ++t)
            if ((pending >> t) & 1u) mbar_wait(&bar[t], (parity >> t) & 1u);
    }
}

template <class IT, class V, bool NUMERIC, class K>
cudaError_t merge_grid(K k, long long units, int sm_count, size_t* smem, unsigned* grid) {
    *smem = (size_t)kMergeWarps * MergeWarp<V, NUMERIC>::kBytes;
    if (*smem > 48 * 1024) {
        cudaError_t e =
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)*smem);
        if (e != cudaSuccess) return e;
    }
    int occ = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, kMergeWarps * 32, *smem);
    if (occ < 1) occ = 1;
    *grid = (unsigned)std::max<long long>(
        1, std::min((units + kMergeWarps - 1) / kMergeWarps, (long long)sm_count * occ));
    return cudaSuccess;
}

template <class IT, class V, bool NUMERIC>
cudaError_t launch_merge_segments(int c, const MergeParts<IT, V>& mp, int sm_count,
                                  cudaStream_t s, int64_t* rowcnt, const int64_t* rpC, IT* colC,
                                  V* valC, int* err, MergeLong* longs) {
    auto k = merge_segments_kernel<IT, V, NUMERIC>;
    size_t smem = 0;
    unsigned g = 1;
    cudaError_t e = merge_grid<IT, V, NUMERIC>(k, (long long)kMergeLongRows * kMergeSegs, sm_count,
                                               &smem, &g);
    if (e != cudaSuccess) return e;
    count_launches(1);
    k<<<g, kMergeWarps * 32, smem, s>>>(c, mp, rowcnt, rpC, colC, valC, err,
                                        &longs->work[NUMERIC ? 1 : 0], longs);
    return cudaGetLastError();
}

template <class IT, class V, bool NUMERIC>
cudaError_t launch_merge_t(int c, const spgemm_csr* parts, long long m, long long n,
                           int sm_count, cudaStream_t s, int64_t* rowcnt, const int64_t* rpC,
                           void* colC, void* valC, int* err, unsigned long long* work,
                           MergeLong* longs, bool staged_opt) {
    if (m <= 0) return cudaSuccess;
    MergeParts<IT, V> mp{};
    long long entries = 0;   // at most: a part's arrays may hold more than its rows
    for (int t = 0; t < c; ++t) {
        mp.rp[t] = parts[t].rowptr;
        mp.re[t] = parts[t].rowend;
        mp.col[t] = (const IT*)parts[t].col;
        mp.val[t] = (const V*)parts[t].val;
        mp.len[t] = parts[t].nnz;
        entries += parts[t].nnz;
    }
    if constexpr (NUMERIC) {
        bool staged = staged_opt && c <= 4;
        for (int t = 0; t < c; ++t)
            staged = staged && ((uintptr_t)parts[t].col % 16) == 0 &&
                     (!VOps<V>::has_val || ((uintptr_t)parts[t].val % 16) == 0);
        if (staged) {
            constexpr int W = 1024, WARPS = 4, WIN = 64;
            auto k = c <= 2 ? merge_stage_kernel<IT, V, W, WARPS, 2, WIN>
                            : merge_stage_kernel<IT, V, W, WARPS, 4, WIN>;
            const size_t smem = (size_t)WARPS * (c <= 2 ? MergeStage<IT, V, W, WARPS, 2, WIN>::warp_bytes
                                                          : MergeStage<IT, V, W, WARPS, 4, WIN>::warp_bytes);
            if (smem > 48 * 1024) {
                cudaError_t e =
                    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
                if (e != cudaSuccess) return e;
            }
            int occ = 1;
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, WARPS * 32, smem);
            if (occ < 1) occ = 1;
            const long long need = (m + WARPS - 1) / WARPS;
            const long long g = std::max<long long>(1, std::min(need, (long long)sm_count * occ));
            count_launches(1);
            k<<<(unsigned)g, WARPS * 32, smem, s>>>(c, mp, m, n, rpC, (IT*)colC, (V*)valC, err, work);
            return cudaGetLastError();
        }
    }
    if (entries <= kMergeLong) longs = nullptr;   // no row can be long
    cudaError_t e;
    if (longs && (e = cudaMemsetAsync(longs, 0, kMergeLongHead, s)) != cudaSuccess) return e;
    auto k = merge_rows_kernel<IT, V, NUMERIC>;
    size_t smem = 0;
    unsigned g = 1;
    if ((e = merge_grid<IT, V, NUMERIC>(k, m, sm_count, &smem, &g)) != cudaSuccess) return e;
    count_launches(1);
    k<<<g, kMergeWarps * 32, smem, s>>>(c, mp, m, rowcnt, rpC, (IT*)colC, (V*)valC, err, work, longs);
    if ((e = cudaGetLastError()) != cudaSuccess || !longs) return e;
    // the listed rows' segments: counted, and for the numeric pass then filled
    e = launch_merge_segments<IT, V, false>(c, mp, sm_count, s, NUMERIC ? nullptr : rowcnt,
                                            nullptr, nullptr, nullptr, err, longs);
    if constexpr (NUMERIC)
        if (e == cudaSuccess)
            e = launch_merge_segments<IT, V, true>(c, mp, sm_count, s, nullptr, rpC, (IT*)colC,
                                                   (V*)valC, err, longs);
    return e;
}

cudaError_t launch_merge(int c, const spgemm_csr* parts, int vt, long long m, long long n,
                         int sm_count, cudaStream_t s, bool numeric, int64_t* rowcnt,
                         const int64_t* rpC, void* colC, void* valC, int* err,
                         unsigned long long* work, MergeLong* longs, bool staged) {
    const bool i32 = parts[0].index_type == SPGEMM_INDEX_I32;
    return with_value_type(vt, [&](auto tag) -> cudaError_t {
        using V = decltype(tag);
        if (numeric)
            return i32 ? launch_merge_t<int32_t, V, true>(c, parts, m, n, sm_count, s, rowcnt, rpC,
                                                          colC, valC, err, work, longs, staged)
                       : launch_merge_t<int64_t, V, true>(c, parts, m, n, sm_count, s, rowcnt, rpC,
                                                          colC, valC, err, work, longs, staged);
        return i32 ? launch_merge_t<int32_t, V, false>(c, parts, m, n, sm_count, s, rowcnt, rpC,
                                                       colC, valC, err, work, longs, staged)
                   : launch_merge_t<int64_t, V, false>(c, parts, m, n, sm_count, s, rowcnt, rpC,
                                                       colC, valC, err, work, longs, staged);
    });
}

}  // namespace sg
