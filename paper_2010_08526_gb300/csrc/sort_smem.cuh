// Sorted compaction of a shared-memory hash table: the paper keeps the final
// C sorted within its columns (Sec. IV-D), so a column (or work item) that
// was accumulated in a table leaves it in row order, without a second pass
// over the output.
//
// A table of T slots holds n <= T / 2 entries. They are moved to the front of
// the table, which frees its upper half as scratch, and ordered there:
//   1. buckets: row - lowest row, shifted so that the span fits NB = T / 4
//      buckets (a counting sort on the leading bits; rows are distinct, so a
//      bucket holds at most 2^shift of them);
//   2. each entry's place inside its bucket by counting the smaller rows of
//      the bucket (one or two on average; neighbouring lanes mostly read the
//      same bucket, so the loads broadcast);
//   3. the write, whose lanes go to neighbouring places: coalesced stores.
// The work is O(n) for spread-out rows. Clusters that overfill a bucket
// (kSortMaxBucket, kSortMaxBucketWarp) fall back to the bitonic network over the
// front entries.
//
// It takes the place of a bitonic sort of the written output in a kernel of
// its own (two more passes over C, 91 barrier-separated stages at 8192
// entries). Measured: the protein stand-in with 100,000 columns (int64 / fp32,
// 5.3e8 entries) spent 26.4 ms in those kernels and spends 0.95 ms more in the
// CTA tiers now (step 40.3 -> 14.8 ms); R-MAT scale 14 fp32 4.1 -> 0.15 ms
// (6.8 -> 3.0 ms); 2-path counts of a 50,021-vertex uniform graph 1.13 -> 0.07 ms.
#pragma once

namespace spg {

// The group working on one table: a whole CTA, or one warp (ss unused).
template <bool BLOCK> __device__ __forceinline__ void sort_sync() {
    if constexpr (BLOCK) __syncthreads(); else __syncwarp();
}

// Bitonic sort of n entries in shared memory by the group (keys padded with
// 0xffffffff to the next power of two). All its threads call it.
template <bool BLOCK, class V>
__device__ __forceinline__ void bitonic(uint32_t *sk, V *sv, int n) {
    const int t = BLOCK ? (int)threadIdx.x : (int)(threadIdx.x & 31), nt = BLOCK ? (int)blockDim.x : 32;
    int np2 = 1;
    while (np2 < n) np2 <<= 1;
    for (int i = n + t; i < np2; i += nt) { sk[i] = 0xffffffffu; sv[i] = V(0); }
    sort_sync<BLOCK>();
    for (int k = 2; k <= np2; k <<= 1) {
        for (int jj = k >> 1; jj > 0; jj >>= 1) {
            for (int p = t; p < np2 / 2; p += nt) {   // pair p: entries i and i + jj
                const int i = ((p & ~(jj - 1)) << 1) | (p & (jj - 1)), l = i | jj;
                const bool up = (i & k) == 0;
                const uint32_t a = sk[i], b = sk[l];
                if (up ? a > b : a < b) {
                    sk[i] = b; sk[l] = a;
                    const V x = sv[i]; sv[i] = sv[l]; sv[l] = x;
                }
            }
            sort_sync<BLOCK>();
        }
    }
}

// The warp's network as a call: inlined, it spills the walks around it (k_light with
// 256 int64 slots 28 -> 140 bytes, 2-path counts of 50,021 vertices 463 -> 485 us).
template <class V> __device__ __noinline__ void bitonic_warp(uint32_t *sk, V *sv, int n) { bitonic<false>(sk, sv, n); }

// A bucket above this many entries sends a CTA's (a warp's) table to the bitonic
// sort: counting costs a bucket its square. Columns of clusters of consecutive rows far
// apart, ranked however full a bucket is (up to 512 in a CTA) -> with these lines,
// fp32, times an identity: 1 x 500 rows (40,000 columns, a warp each) 1.86 -> 0.80 ms, 1 x 250
// (80,000) 0.96 -> 0.73, 2 x 500 (20,000, a CTA each) 1.65 -> 1.03, 8 x 500 (6,000) 2.02 -> 1.59;
// 128 in a CTA loses (16 x 250 rows 1.24 against 1.65 ms), and so does 64 in a warp (1 x 90
// rows 0.71 against 0.92).
constexpr int kSortMaxBucket = 256;
constexpr int kSortMaxBucketWarp = 128;

// CTA-wide scratch of the sorted compaction (a warp needs none)
struct SortShared {
    int n;               // entries compacted so far
    uint32_t lo, hi;     // span of their rows
    int most;            // fullest bucket
    int red[33];
};

// To be called (followed by a barrier) before each sort_front of a CTA that
// did not go through compact_front.
__device__ __forceinline__ void sort_reset(SortShared *ss) {
    ss->n = 0; ss->lo = 0xffffffffu; ss->hi = 0u; ss->most = 0;
}

// Moves the occupied slots of a table to its front; returns their number
// and this thread's span of rows in lo, hi. BLOCK: sort_reset(ss) and a
// barrier come first. Ends before the last writes are visible to the group.
// In place: a round reads four slots per thread, and what it writes lies
// below every slot that a later round reads.
template <bool BLOCK, class V>
__device__ __forceinline__ int compact_front(uint32_t *keys, V *vals, int T, SortShared *ss, uint32_t &lo,
                                             uint32_t &hi) {
    const int lane = threadIdx.x & 31;
    const int t = BLOCK ? (int)threadIdx.x : lane, nt = BLOCK ? (int)blockDim.x : 32;
    const unsigned below = (1u << lane) - 1u;
    int n = 0;
    lo = 0xffffffffu;
    hi = 0u;
    for (int s0 = 0; s0 < T; s0 += 4 * nt) {
        uint32_t k[4];
        V v[4];
        unsigned bal[4];
        int c = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int s = s0 + u * nt + t;
            k[u] = s < T ? keys[s] : kEmpty;
            if (k[u] != kEmpty) v[u] = vals[s];
            bal[u] = __ballot_sync(SPG_FULL, k[u] != kEmpty);
            c += __popc(bal[u]);
        }
        int base = n;
        if constexpr (BLOCK) {
            if (lane == 0 && c) base = atomicAdd(&ss->n, c);
            base = __shfl_sync(SPG_FULL, base, 0);
        } else {
            n += c;
        }
        sort_sync<BLOCK>();   // every slot of the round has been read
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (k[u] != kEmpty) {
                const int at = base + __popc(bal[u] & below);
                keys[at] = k[u];
                vals[at] = v[u];
                lo = min(lo, k[u]);
                hi = max(hi, k[u]);
            }
            base += __popc(bal[u]);
        }
    }
    if constexpr (BLOCK) n = ss->n;   // final after the last round's barrier
    return n;
}

// Writes the n <= T / 2 front entries of a table in row order (want: the
// exact count, the number of output places). lo, hi: each thread's span of
// rows. The upper half of the table is scratch. T is a power of two >= 64.
template <bool BLOCK, class V, class I>
__device__ __forceinline__ void sort_front(uint32_t *keys, V *vals, int T, int n, uint32_t lo, uint32_t hi,
                                           int want, SortShared *ss, I *out_rows, V *out_vals) {
    const int lane = threadIdx.x & 31;
    const int t = BLOCK ? (int)threadIdx.x : lane, nt = BLOCK ? (int)blockDim.x : 32;
    const int cap = T >> 1, NB = T >> 2;
    if (!BLOCK && n <= 32) {
        // one entry per lane: its place is the number of smaller rows
        __syncwarp();
        const uint32_t key = lane < n ? keys[lane] : kEmpty;
        int r = 0;
        for (int j = 0; j < n; ++j) r += keys[j] < key;
        if (lane < n && r < want) { out_rows[r] = (I)key; out_vals[r] = vals[lane]; }
        return;
    }
    uint32_t *skey = keys + cap;                                   // rows in bucket order
    uint32_t *hist = reinterpret_cast<uint32_t *>(vals + cap);     // NB bucket counts, then their ends
    uint16_t *sidx = reinterpret_cast<uint16_t *>(hist + NB);      // front position of skey[i]
    lo = __reduce_min_sync(SPG_FULL, lo);
    hi = __reduce_max_sync(SPG_FULL, hi);
    if constexpr (BLOCK) {
        if (lane == 0) { atomicMin(&ss->lo, lo); atomicMax(&ss->hi, hi); }
    }
    sort_sync<BLOCK>();   // the front is complete: the upper half is free
    for (int i = t; i < NB / 4; i += nt) reinterpret_cast<uint4 *>(hist)[i] = make_uint4(0u, 0u, 0u, 0u);
    if constexpr (BLOCK) { lo = ss->lo; hi = ss->hi; }
    const int bits = 32 - __clz((int)(hi - lo));      // of the span (0: a single row)
    const int shift = max(0, bits - (31 - __clz(NB)));
    sort_sync<BLOCK>();
    for (int i = t; i < n; i += nt) atomicAdd(&hist[(keys[i] - lo) >> shift], 1u);
    sort_sync<BLOCK>();
    // exclusive prefix of the bucket counts, a run of buckets (in fours) per thread
    uint4 *hist4 = reinterpret_cast<uint4 *>(hist);
    const int per = (NB / 4 + nt - 1) / nt;
    const int b0 = min(NB / 4, t * per), b1 = min(NB / 4, b0 + per);
    int sum = 0;
    uint32_t most = 0;
    for (int b = b0; b < b1; ++b) {
        const uint4 c = hist4[b];
        sum += (int)(c.x + c.y + c.z + c.w);
        most = max(most, max(max(c.x, c.y), max(c.z, c.w)));
    }
    const int incl = warp_incl_scan(sum);
    int run = incl - sum;
    if constexpr (BLOCK) {
        const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
        most = __reduce_max_sync(SPG_FULL, most);
        if (lane == 31) ss->red[warp] = incl;
        if (lane == 0 && shift > 8) atomicMax(&ss->most, (int)most);   // at most 2^shift per bucket
        __syncthreads();
        const int w = lane < nw ? ss->red[lane] : 0;
        const int wi = warp_incl_scan(w);
        run += __shfl_sync(SPG_FULL, wi - w, warp);
        if (ss->most > kSortMaxBucket) {   // the same for the whole CTA
            bitonic<true>(keys, vals, n);
            for (int i = t; i < n && i < want; i += nt) { out_rows[i] = (I)keys[i]; out_vals[i] = vals[i]; }
            return;
        }
    } else if (cap > kSortMaxBucketWarp && shift > 7) {   // likewise; cap is the caller's constant
        most = __reduce_max_sync(SPG_FULL, most);
        if (most > kSortMaxBucketWarp) {   // the same for the warp
            bitonic_warp(keys, vals, n);
            for (int i = t; i < n && i < want; i += nt) { out_rows[i] = (I)keys[i]; out_vals[i] = vals[i]; }
            return;
        }
    }
    for (int b = b0; b < b1; ++b) {
        const uint4 c = hist4[b];
        const uint32_t x = (uint32_t)run, y = x + c.x, z = y + c.y, w = z + c.z;
        hist4[b] = make_uint4(x, y, z, w);
        run = (int)(w + c.w);
    }
    sort_sync<BLOCK>();
    for (int i = t; i < n; i += nt) {
        const uint32_t key = keys[i];
        const uint32_t at = atomicAdd(&hist[(key - lo) >> shift], 1u);
        skey[at] = key;
        sidx[at] = (uint16_t)i;
    }
    sort_sync<BLOCK>();   // hist[b] is now the end of bucket b
    for (int i = t; i < n; i += nt) {
        const uint32_t key = skey[i];
        const uint32_t b = (key - lo) >> shift;
        const int e = (int)hist[b];
        int s = b ? (int)hist[b - 1] : 0;
        int r = s;
        for (; s < e; ++s) r += skey[s] < key;
        if (r < want) { out_rows[r] = (I)key; out_vals[r] = vals[sidx[i]]; }
    }
}

// Compacts a table and writes its entries in row order at out_rows /
// out_vals, then leaves every slot empty. A count other than want sets
// kErrCount. BLOCK: all threads call it, after a barrier that ends the
// insertions; it ends with a barrier.
template <bool BLOCK, class V, class I>
__device__ __forceinline__ void sorted_emit(uint32_t *keys, V *vals, int T, int want, SortShared *ss, int *err,
                                            I *out_rows, V *out_vals) {
    const int lane = threadIdx.x & 31;
    const int t = BLOCK ? (int)threadIdx.x : lane, nt = BLOCK ? (int)blockDim.x : 32;
    if constexpr (BLOCK) {
        if (threadIdx.x == 0) sort_reset(ss);
        __syncthreads();
    }
    uint32_t lo, hi;
    const int n = compact_front<BLOCK>(keys, vals, T, ss, lo, hi);
    if (n != want && t == 0) atomicOr(err, kErrCount);
    if (n <= (T >> 1)) sort_front<BLOCK>(keys, vals, T, n, lo, hi, want, ss, out_rows, out_vals);
    sort_sync<BLOCK>();
    // empty slots again, 16 bytes at a time (tables start on 16-byte boundaries)
    uint4 *k4 = reinterpret_cast<uint4 *>(keys);
    struct alignas(16) Vals { V v[16 / sizeof(V)]; };
    Vals *v4 = reinterpret_cast<Vals *>(vals);
    Vals none;
#pragma unroll
    for (int i = 0; i < 16 / (int)sizeof(V); ++i) none.v[i] = V(0);
    for (int s = t; s < T / 4; s += nt) k4[s] = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
    for (int s = t; s < T * (int)sizeof(V) / 16; s += nt) v4[s] = none;
    sort_sync<BLOCK>();
}

}  // namespace spg
