// Sorted final output and the column-wise prune of a result batch.
//
// Sorting: the paper keeps the final C sorted within each column (Sec. IV-D:
// only the intermediate products are left unsorted). The numeric kernels write
// row order themselves (sort_smem.cuh, dense items by nature). Two sorts of
// written output remain: the hash-range items of heavy columns where the generic
// heavy kernel made them (the merge, nnz(A) >= 2^31 - 8192; k_sort_items), and the pruned
// columns of a batch (k_sort_cols).
//
// Prune: the consumer the column batches are shaped for keeps the largest
// entries of every column (Markov clustering, Sec. III; HipMCL prunes each
// batch, Sec. V-F). Per column: candidates are the entries with value >=
// threshold; if topk > 0 and more remain, the topk largest are kept, equal
// values going to the earlier stored entry; kept entries stay in their order.
#pragma once

#include <type_traits>

#include "kernels.cuh"

namespace spg {

// ---- order-preserving keys ------------------------------------------------
// Unsigned keys whose order is the order of the values (IEEE floats: the sign
// bit flipped for positives, all bits flipped for negatives; int64: the sign
// bit flipped). NaN never reaches them: it fails every threshold test.
__device__ __forceinline__ uint64_t value_key(float v) {
    const uint32_t u = __float_as_uint(v);
    return (uint64_t)(u ^ ((u >> 31) ? 0xffffffffu : 0x80000000u));
}
__device__ __forceinline__ uint64_t value_key(double v) {
    const uint64_t u = (uint64_t)__double_as_longlong(v);
    return u ^ ((u >> 63) ? 0xffffffffffffffffull : 0x8000000000000000ull);
}
__device__ __forceinline__ uint64_t value_key(int64_t v) { return (uint64_t)v ^ 0x8000000000000000ull; }
template <class F> __device__ __forceinline__ uint64_t value_key(MinPlus<F> v) { return value_key(v.v); }
template <class T> __device__ __forceinline__ uint64_t value_key(OrAnd<T> v) { return value_key(v.v); }
template <class V> struct KeyBits { static constexpr int v = 64; };
template <> struct KeyBits<float> { static constexpr int v = 32; };
template <> struct KeyBits<MinPlus<float>> { static constexpr int v = 32; };
template <> struct KeyBits<OrAnd<float>> { static constexpr int v = 32; };

// ---- sort ------------------------------------------------------------------
// Sorts the columns with lo_excl < n <= T / 2 entries in place, through a table
// of T slots in shared memory (sort_front): one warp per column, or one CTA
// for the larger tables. colptr is relative (columns [0, ncols)).
template <class I, class V, int T, bool BLOCK>
__global__ void __launch_bounds__(BLOCK ? 512 : 256) k_sort_cols(const int64_t *colptr, int64_t ncols, int lo_excl,
                                                                 I *rows, V *vals) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ SortShared ss;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int nt = BLOCK ? (int)blockDim.x : 32, t = BLOCK ? (int)threadIdx.x : lane;
    const int tables = BLOCK ? 1 : nw;
    V *sv = reinterpret_cast<V *>(smem) + (BLOCK ? 0 : warp * T);
    uint32_t *sk = reinterpret_cast<uint32_t *>(smem + sizeof(V) * tables * T) + (BLOCK ? 0 : warp * T);
    const int64_t step = BLOCK ? gridDim.x : (int64_t)gridDim.x * nw;
    for (int64_t j = BLOCK ? blockIdx.x : (int64_t)blockIdx.x * nw + warp; j < ncols; j += step) {
        const int64_t a = colptr[j];
        const int64_t n64 = colptr[j + 1] - a;
        if (n64 <= lo_excl || n64 > T / 2 || n64 < 2) continue;
        const int n = (int)n64;
        uint32_t lo = 0xffffffffu, hi = 0u;
        if (BLOCK && threadIdx.x == 0) sort_reset(&ss);
        for (int i = t; i < n; i += nt) {
            const uint32_t r = (uint32_t)rows[a + i];
            sk[i] = r;
            sv[i] = vals[a + i];
            lo = min(lo, r);
            hi = max(hi, r);
        }
        sort_sync<BLOCK>();
        sort_front<BLOCK>(sk, sv, T, n, lo, hi, n, &ss, rows + a, vals + a);
        sort_sync<BLOCK>();
    }
}

// One CTA per hash-range item of a heavy column in [c0, c1). The item's
// rows are distinct and lie in its row range [p0 R, p1 R), so a bitmap over
// the range ranks them: set a bit per row, prefix the word popcounts, and an
// entry's position is the number of set bits below its row. O(n + range/32)
// per item. A range wider than the bitmap words given (wcap) falls back to
// the bitonic sort. Dense items are in row order already.
template <class I, class V, int CAP>
__global__ void __launch_bounds__(512, 2) k_sort_items(const HeavyItem *items, const int64_t *nitems_p, const int64_t *colptr,
                             int64_t base, int64_t c0, int64_t c1, int log2R, int wcap, I *rows, V *vals) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t *sk = reinterpret_cast<uint32_t *>(smem);                       // CAP staged rows
    V *sv = reinterpret_cast<V *>(smem + sizeof(uint32_t) * CAP);            // CAP staged values
    uint32_t *bm = reinterpret_cast<uint32_t *>(smem + (sizeof(uint32_t) + sizeof(V)) * CAP);
    uint16_t *pre = reinterpret_cast<uint16_t *>(bm + wcap);                 // word prefix (< CAP <= 2^15)
    __shared__ uint32_t s_part[1024];
    const int64_t nitems = *nitems_p;
    for (int64_t it = blockIdx.x; it < nitems; it += gridDim.x) {
        const HeavyItem item = items[it];
        if (item.cnt <= 1 || item.cnt > CAP || item.g < c0 || item.g >= c1) continue;   // dense (< 0) or trivial
        const int n = item.cnt;
        const int64_t a = colptr[item.g] - base + item.off;
        const int64_t r0 = (int64_t)item.p0 << log2R;
        const int W = (int)((((int64_t)(item.p1 - item.p0)) << log2R) >> 5);
        if (W > wcap) {
            for (int i = threadIdx.x; i < n; i += blockDim.x) { sk[i] = (uint32_t)rows[a + i]; sv[i] = vals[a + i]; }
            bitonic<true>(sk, sv, n);
            for (int i = threadIdx.x; i < n; i += blockDim.x) { rows[a + i] = (I)sk[i]; vals[a + i] = sv[i]; }
            __syncthreads();
            continue;
        }
        for (int w = threadIdx.x; w < W; w += blockDim.x) bm[w] = 0u;
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            const uint32_t r = (uint32_t)rows[a + i];
            sk[i] = r;
            sv[i] = vals[a + i];
            const uint32_t b = (uint32_t)((int64_t)r - r0);
            atomicOr(&bm[b >> 5], 1u << (b & 31));
        }
        __syncthreads();
        // exclusive prefix of the word popcounts: each thread a contiguous
        // run of words, then a scan over the threads' sums
        const int per = (W + (int)blockDim.x - 1) / (int)blockDim.x;
        const int w0 = threadIdx.x * per, w1 = min(W, w0 + per);
        uint32_t sum = 0;
        for (int w = w0; w < w1; ++w) sum += __popc(bm[w]);
        s_part[threadIdx.x] = sum;
        __syncthreads();
        for (int o = 1; o < (int)blockDim.x; o <<= 1) {
            const uint32_t t = threadIdx.x >= (unsigned)o ? s_part[threadIdx.x - o] : 0u;
            __syncthreads();
            s_part[threadIdx.x] += t;
            __syncthreads();
        }
        uint32_t run = s_part[threadIdx.x] - sum;
        for (int w = w0; w < w1; ++w) { pre[w] = (uint16_t)run; run += __popc(bm[w]); }
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            const uint32_t b = (uint32_t)((int64_t)sk[i] - r0);
            const uint32_t pos = (uint32_t)pre[b >> 5] + __popc(bm[b >> 5] & ((1u << (b & 31)) - 1u));
            rows[a + pos] = (I)sk[i];
            vals[a + pos] = sv[i];
        }
        __syncthreads();
    }
}

// int32 colptr widened to int64
template <class T>
__global__ void k_widen(const T *src, int64_t n, int64_t *dst) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = (int64_t)src[i];
}

// ---- prune -----------------------------------------------------------------
// Per column j of a batch (colptr relative offsets, ncols columns):
// keep[j] = kept count; a column that needs a selection (more candidates than
// topk) goes to sel_list. mode[j]: 0 keep every candidate, 1 selection. A warp
// per column with four loads in flight per lane.
template <class V>
__global__ void __launch_bounds__(256) k_prune_count(const int64_t *colptr, const V *vals, int64_t ncols,
                                                     V thr, int64_t topk, int64_t *keep, int8_t *mode,
                                                     int64_t *sel_list, unsigned long long *nsel) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; j < ncols; j += nw) {
        const int64_t a = colptr[j] - colptr[0], b = colptr[j + 1] - colptr[0];
        int64_t c = 0;
        int64_t q = a + lane;
        for (; q + 96 < b; q += 128) {
            const V x0 = vals[q], x1 = vals[q + 32], x2 = vals[q + 64], x3 = vals[q + 96];
            c += (x0 >= thr) + (x1 >= thr) + (x2 >= thr) + (x3 >= thr);
        }
        for (; q < b; q += 32) c += vals[q] >= thr;
        c = warp_sum(c);
        if (lane == 0) {
            if (topk > 0 && c > topk) {
                keep[j] = topk;
                mode[j] = 1;
                sel_list[atomicAdd(nsel, 1ull)] = j;
            } else {
                keep[j] = c;
                mode[j] = 0;
            }
        }
    }
}

// Unsigned keys of the value's own width, whose order is the values' (see
// value_key); a value below the threshold, or NaN, gets a key below cand_key().
template <int BITS> struct KeyOf { using type = uint64_t; };
template <> struct KeyOf<32> { using type = uint32_t; };
template <class V> struct IsIntValue { static constexpr bool v = std::is_integral<typename Storage<V>::type>::value; };
// no candidate has key 0 for floats (the all-ones NaN); integers keep their keys
template <class V, class K> __device__ __forceinline__ K cand_key(V thr) {
    return IsIntValue<V>::v ? (K)value_key(thr) : (K)1;
}
template <class V, class K> __device__ __forceinline__ K prune_key(V v, V thr) {
    return IsIntValue<V>::v || v >= thr ? (K)value_key(v) : (K)0;
}

constexpr int kPruneThreads = 512;

// One CTA per listed column (nsel[0] of them, taken through nsel[1]): finds the topk-th largest key among the
// candidates and writes the kept entries, in stored order, at out_colptr[j].
// The selection is a radix select, 8 bits a pass, on the key's distance from
// the column's smallest candidate: the leading equal bits (sign, exponent) are
// skipped, and the digits spread over the bins instead of crowding into a few.
// Keys are staged in shared memory when the column fits (cap), so the
// passes read the values from memory once.
// Places in a column are unsigned 32-bit numbers: a column has fewer than 2^31 entries, and
// the passes step past its end.
// Equal keys at the cut: the earlier stored ones are kept, or (tie_by_row != 0)
// the smaller rows, found by a second select over the ties' rows.
// Measured (protein stand-in, 20,011 columns in 4 batches, top 100): counting,
// selecting and compacting in three kernels, the last a warp per column with one
// load in flight, took 1.88 ms, this and the count 0.93 ms (three CTAs per SM: 1.08 ms, the registers spill).
template <class I, class V, class IO>
__global__ void __launch_bounds__(kPruneThreads, 2) k_prune_select(const int64_t *colptr, const I *rows, const V *vals,
                                                                V thr, int64_t topk, const int64_t *sel_list,
                                                                unsigned long long *nsel, int tie_by_row, int cap,
                                                                const int64_t *out_colptr, IO *out_rows,
                                                                V *out_vals) {
    using K = typename KeyOf<KeyBits<V>::v>::type;
    constexpr int NW = kPruneThreads / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    K *sk = reinterpret_cast<K *>(smem);
    __shared__ uint32_t hist[4][256];
    __shared__ K s_min[NW], s_max[NW];
    __shared__ int s_digit;
    __shared__ uint32_t s_k, s_in;
    __shared__ int s_hi[NW], s_tie[NW];
    __shared__ long long s_item;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    const int64_t ns = (int64_t)*nsel;
    const K ck = cand_key<V, K>(thr);

    // the digit (highest bin for keys, lowest for rows) at which the count
    // from the top (bottom) reaches k: s_digit, s_k = what remains of k in it,
    // s_in = entries in it. All threads call it.
    auto pick = [&](uint32_t k, bool from_top) {
        __syncthreads();
        if (warp == 0) {
            uint32_t c8[8], mine = 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int bin = from_top ? 255 - (lane * 8 + i) : lane * 8 + i;
                c8[i] = hist[0][bin] + hist[1][bin] + hist[2][bin] + hist[3][bin];
                mine += c8[i];
            }
            uint32_t acc = warp_incl_scan(mine) - mine;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (acc < k && acc + c8[i] >= k) {   // one lane and bin
                    s_digit = from_top ? 255 - (lane * 8 + i) : lane * 8 + i;
                    s_k = k - acc;
                    s_in = c8[i];
                }
                acc += c8[i];
            }
        }
        __syncthreads();
    };
    auto clear_hist = [&]() {
        for (int i = threadIdx.x; i < 4 * 256; i += kPruneThreads) (&hist[0][0])[i] = 0u;
        __syncthreads();
    };

    for (;;) {
        // columns differ in length: taken from a device counter
        if (threadIdx.x == 0) s_item = (long long)atomicAdd(nsel + 1, 1ull);
        __syncthreads();
        const int64_t s = s_item;
        if (s >= ns) break;
        const int64_t j = sel_list[s];
        const int64_t a = colptr[j] - colptr[0];
        const uint32_t n = (uint32_t)(colptr[j + 1] - colptr[j]);
        const bool staged = n <= (uint32_t)cap;
        auto key_at = [&](uint32_t i) -> K { return staged ? sk[i] : prune_key<V, K>(vals[a + i], thr); };
        // every key of the column, four loads in flight per thread
        auto each = [&](auto &&f) {
            for (uint32_t i0 = threadIdx.x; i0 < n; i0 += 4 * kPruneThreads) {
                K x[4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    x[u] = i0 + u * kPruneThreads < n ? key_at(i0 + u * kPruneThreads) : (K)0;
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (i0 + u * kPruneThreads < n && x[u] >= ck) f(i0 + u * kPruneThreads, x[u]);
            }
        };
        // keys and their span
        K lo = ~K(0), hi = 0;
        for (uint32_t i0 = threadIdx.x; i0 < n; i0 += 4 * kPruneThreads) {
            V v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (i0 + u * kPruneThreads < n) v[u] = vals[a + i0 + u * kPruneThreads];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + u * kPruneThreads;
                if (i >= n) break;
                const K k = prune_key<V, K>(v[u], thr);
                if (staged) sk[i] = k;
                if (k >= ck) { lo = min(lo, k); hi = max(hi, k); }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo = min(lo, (K)__shfl_xor_sync(SPG_FULL, lo, o));
            hi = max(hi, (K)__shfl_xor_sync(SPG_FULL, hi, o));
        }
        if (lane == 0) { s_min[warp] = lo; s_max[warp] = hi; }
        __syncthreads();
#pragma unroll
        for (int w = 0; w < NW; ++w) { lo = min(lo, s_min[w]); hi = max(hi, s_max[w]); }
        // radix select on key - lo; rb: bits below the ones decided
        int rb = hi == lo ? 0 : 64 - __clzll((long long)(uint64_t)(hi - lo));
        K prefix = 0;
        uint32_t k = (uint32_t)topk;
        bool whole = false;   // every entry of the selected bin is kept
        while (rb > 0) {
            const int w = min(8, rb), sh = rb - w;
            clear_hist();
            const bool first = rb == (int)sizeof(K) * 8;   // a shift by the whole width is undefined
            each([&](uint32_t, K key) {
                const K d = key - lo;
                if (!first && (K)(d >> rb) != prefix) return;
                atomicAdd(&hist[warp & 3][(uint32_t)(d >> sh) & ((1u << w) - 1u)], 1u);
            });
            pick(k, true);
            prefix = (K)((prefix << w) | (K)s_digit);
            k = s_k;
            whole = s_in == k;
            rb = sh;
            if (whole) break;   // the same for the whole CTA
        }
        // kept: (key - lo) >> rb above prefix, and k of those equal to it
        uint32_t rmax = 0xffffffffu;
        if (!whole && tie_by_row) {
            // the k-th smallest row among the ties (rows are distinct)
            uint32_t rpre = 0, rk = k;
            for (int sh = 24; sh >= 0; sh -= 8) {
                clear_hist();
                each([&](uint32_t i, K key) {
                    if ((K)((key - lo) >> rb) != prefix) return;
                    const uint32_t r = (uint32_t)rows[a + i];
                    if (sh < 24 && (r >> (sh + 8)) != rpre) return;
                    atomicAdd(&hist[warp & 3][(r >> sh) & 255u], 1u);
                });
                pick(rk, false);
                rpre = (rpre << 8) | (uint32_t)s_digit;
                rk = s_k;
            }
            rmax = rpre;
        }
        // stable compaction: a warp takes 128 consecutive entries of a step
        const int64_t o = out_colptr[j] - out_colptr[0];
        uint32_t done_hi = 0, done_tie = 0;
        for (uint32_t c0 = 0; c0 < n; c0 += 4 * kPruneThreads) {
            const uint32_t i0 = c0 + warp * 128 + lane;
            bool up[4], tie[4];
            int nh = 0, nt = 0;
            unsigned bh[4], bt[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + 32 * u;
                up[u] = tie[u] = false;
                if (i < n) {
                    const K key = key_at(i);
                    if (key >= ck) {
                        const K d = (K)((key - lo) >> rb);
                        up[u] = d > prefix || (d == prefix && whole);
                        tie[u] = d == prefix && !whole;
                    }
                }
                if (tie[u] && tie_by_row) {
                    up[u] = (uint32_t)rows[a + i] <= rmax;
                    tie[u] = false;
                }
                bh[u] = __ballot_sync(SPG_FULL, up[u]);
                bt[u] = __ballot_sync(SPG_FULL, tie[u]);
                nh += __popc(bh[u]);
                nt += __popc(bt[u]);
            }
            if (lane == 0) { s_hi[warp] = nh; s_tie[warp] = nt; }
            __syncthreads();
            const int vh = lane < NW ? s_hi[lane] : 0, vt = lane < NW ? s_tie[lane] : 0;
            const int ih = warp_incl_scan(vh), itl = warp_incl_scan(vt);
            uint32_t h0 = done_hi + __shfl_sync(SPG_FULL, ih - vh, warp);
            uint32_t t0 = done_tie + __shfl_sync(SPG_FULL, itl - vt, warp);
            done_hi += __shfl_sync(SPG_FULL, ih, 31);
            done_tie += __shfl_sync(SPG_FULL, itl, 31);
            // the entries of all four windows are read before any is written
            I r[4];
            V x[4];
            int64_t d[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t tb = t0 + __popc(bt[u] & below);   // ties before this entry
                const int64_t q = a + i0 + 32 * u;
                d[u] = -1;
                if (up[u] || (tie[u] && tb < k)) {
                    d[u] = o + h0 + __popc(bh[u] & below) + min(tb, k);
                    r[u] = __ldg(&rows[q]);
                    x[u] = vals[q];
                }
                h0 += __popc(bh[u]);
                t0 += __popc(bt[u]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (d[u] >= 0) { out_rows[d[u]] = (IO)r[u]; out_vals[d[u]] = x[u]; }
            __syncthreads();
        }
    }
}

// One warp per column that keeps all its candidates: stable compaction into
// the output at out_colptr[j] (relative to out_colptr[0]).
template <class I, class V, class IO>
__global__ void __launch_bounds__(256) k_prune_compact(const int64_t *colptr, const I *rows, const V *vals,
                                                       int64_t ncols, V thr, const int8_t *mode,
                                                       const int64_t *out_colptr, IO *out_rows, V *out_vals) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const uint32_t below = (1u << lane) - 1u;
    for (int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; j < ncols; j += nw) {
        if (mode[j] != 0) continue;
        const int64_t a = colptr[j] - colptr[0], b = colptr[j + 1] - colptr[0];
        int64_t o = out_colptr[j] - out_colptr[0];
        for (int64_t q0 = a; q0 < b; q0 += 128) {
            V v[4];
            I r[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t q = q0 + 32 * u + lane;
                if (q < b) { v[u] = vals[q]; r[u] = rows[q]; }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool take = q0 + 32 * u + lane < b && v[u] >= thr;
                const unsigned kb = __ballot_sync(SPG_FULL, take);
                if (take) {
                    const int64_t d = o + __popc(kb & below);
                    out_rows[d] = (IO)r[u];
                    out_vals[d] = v[u];
                }
                o += __popc(kb);
            }
        }
    }
}

}  // namespace spg
