// One persistent launch per pass of the multi-problem product (many
// independent C_i = A_i B_i, each column formed by Sec. II-C's column
// formula): the symbolic count and the numeric hash accumulation of every
// column of every problem run as work items of a single kernel.
//
// Measured, 64 graphs of 500 to 2000 vertices (25.5 M products), bins / symbolic /
// numeric: 54 / 348 / 575 us before, 10 / 186 / 453 us with the problem of a
// column looked up instead of searched, the symbolic pass's shared memory holding
// keys only (12 CTAs per SM, not 7), numeric tables sized by the exact count, CTA
// items written from per-warp runs of slots, and one barrier-free walk for warp
// and CTA items (walk_entries; the CTA-wide walk alone cost 34 and 27 us more).
//
// Work comes from the tier lists of k_bin_scatter (list, off[t]) through two
// device counters. First the CTA items: the columns above the largest
// shared-memory table (heaviest tier first), then the CTA-sized columns
// (largest first), one per item, taken by whole CTAs (atomicAdd on the first
// counter). Then the warp-sized columns: every warp takes a few columns at
// a time from the second counter, with no barrier between warps. Uneven
// problems so balance across SMs without a host round trip.
//
//   CTA item   : a hash table of 2 * cap(tier) slots in shared memory;
//   warp item  : a warp-private table of 2 * cap(tier) <= 2 * 512 slots;
//   heavy item : a hash table in global memory (2 * min(f_j, m) slots,
//                rounded up to a power of two), reached with global atomics.
#pragma once

namespace spg {

struct MultiQueue {
    const int32_t *list;            // global column ids grouped by tier
    const int32_t *off;             // [kTiers + 1] tier offsets in list
    unsigned long long *counter;    // [0] next CTA item, [1] next warp column (zeroed before each launch)
    const int64_t *gtab_off;        // heavy columns: first slot of the global table
    uint32_t *gkeys;                // global tables: keys
    void *gvals;                    // global tables: values
    int warp_tiers;                 // tiers 1..warp_tiers are warp items (<= kWarpTiers)
};

// Global-memory hash insert (linear probing); returns the slot, -1 when the
// table is full (records kErrProbe).
__device__ __forceinline__ int64_t ghash_insert(uint32_t *keys, int log2T, uint32_t key, bool &is_new,
                                                int *err) {
    const uint32_t mask = (1u << log2T) - 1u;
    uint32_t h = hash_slot(key, log2T);
    is_new = false;
    for (uint32_t probe = 0; probe <= mask; ++probe) {
        const uint32_t cur = keys[h];
        if (cur == key) return h;
        if (cur == kEmpty) {
            const uint32_t old = atomicCAS(&keys[h], kEmpty, key);
            if (old == kEmpty) { is_new = true; return h; }
            if (old == key) return h;
        }
        h = (h + 1) & mask;
    }
    atomicOr(err, kErrProbe);
    return -1;
}

// The same sum in global memory (64-bit integer adds are native there).
template <class V> __device__ __forceinline__ void gatomic_add_v(V *p, V v) {
    if constexpr (std::is_same<V, int64_t>::value)
        atomicAdd(reinterpret_cast<unsigned long long *>(p), static_cast<unsigned long long>(v));
    else atomic_add_v(p, v);
}

// MODE 0: symbolic (count distinct rows into c.cnt[g]); MODE 1: numeric
// (accumulate, write column g at c.colptr[g] - c.out_base, unsorted).
template <class Src, int NT, int MODE>
__global__ void __launch_bounds__(NT, MODE == 0 ? 1536 / NT : 0) k_multi_pass(typename Src::Args sa, TierCommon c, MultiQueue mq,
                                                   typename Src::Idx *out_rows, typename Src::Val *out_vals) {
    using V = typename Src::Val;
    using I = typename Src::Idx;
    constexpr int NW = NT / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ BlockShared<V, NT> sh;
    __shared__ long long s_item;
    __shared__ int64_t s_off[NW][32];   // scratch of walk_entries
    __shared__ V s_bv[MODE == 1 ? NW : 1][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int wt = mq.warp_tiers;
    const int nbig = mq.off[kTiers] - mq.off[wt + 1];
    const int nwarp = mq.off[wt + 1] - mq.off[1];
    const int TW = 2 * tier_cap(wt);   // slots of the largest warp table
    if (threadIdx.x == 0) sh.pos = 0;
    for (;;) {
        if (threadIdx.x == 0) s_item = (long long)atomicAdd(mq.counter, 1ull);
        __syncthreads();
        const long long item = s_item;
        __syncthreads();
        if (item >= nbig) break;
        {
            // one column per CTA, heaviest first (the list is ascending in tier)
            const int64_t g = mq.list[mq.off[kTiers] - 1 - item];
            Src src;
            src.open(sa, g);
            const int64_t m = src.m();
            // the tier's capacity bounds the column's distinct rows
            int64_t bound = 0;
            int t = kTiers - 1;
            while (t > wt + 1 && mq.off[t] > mq.off[kTiers] - 1 - item) --t;
            const bool heavy = t >= kHeavyTier0;
            if (!heavy) bound = tier_cap(t);
            int64_t out0 = 0, want = 0;
            if (MODE == 1) {
                out0 = c.colptr[g] - c.out_base;
                want = c.colptr[g + 1] - c.colptr[g];
            }
            if (!heavy) {
                // the numeric pass knows the exact count
                const int64_t rows = MODE == 1 && want < bound ? want : bound;
                int log2T = 7;
                while ((1ll << log2T) < 2 * rows) ++log2T;
                const int T = 1 << log2T;
                V *vals = reinterpret_cast<V *>(smem);
                uint32_t *keys = reinterpret_cast<uint32_t *>(smem + (MODE == 1 ? sizeof(V) * T : 0));
                uint4 *k4 = reinterpret_cast<uint4 *>(keys);
                for (int s = threadIdx.x; s < T / 4; s += NT) k4[s] = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
                if (MODE == 1)
                    for (int s = threadIdx.x; s < T; s += NT) vals[s] = V(0);
                __syncthreads();
                // the warps share a column by rounds of B entries when there are
                // enough of them, else by windows of each round's stream
                int mine = 0;
                auto insert = [&](uint32_t r, V x) {
                    bool nw;
                    const int h = hash_insert_dbl1(keys, log2T, r, c.err, nw);
                    if (MODE == 0) mine += nw;
                    else if (h >= 0) atomic_add_v(&vals[h], x);
                };
                const bool rounds = src.nb >= 64 * NW;
                walk_entries<MODE>(src.p, 0, INT64_MAX, src.b0, (int)src.nb, rounds ? warp : 0, rounds ? NW : 1, rounds ? 0 : warp,
                                   rounds ? 1 : NW, s_off[warp], s_bv[MODE == 1 ? warp : 0], insert);
                __syncthreads();
                if (MODE == 0) {
                    mine = warp_sum(mine);
                    if (lane == 0) sh.red[warp] = mine;
                    __syncthreads();
                    if (threadIdx.x < 32) {
                        int v = threadIdx.x < NW ? sh.red[threadIdx.x] : 0;
                        v = warp_sum(v);
                        if (threadIdx.x == 0) c.cnt[g] = v;
                    }
                } else {
                    // a warp owns a run of slots: count, one barrier, write
                    const int per = (T + NW - 1) / NW;
                    const int slo = min(T, warp * per), shi = min(T, slo + per);
                    int n = 0;
                    for (int s = slo + lane; s < shi; s += 32) n += keys[s] != kEmpty;
                    n = warp_sum(n);
                    int o = warp_offset(n, sh.red, warp, NW, lane);
                    for (int s0 = slo; s0 < shi; s0 += 32) {
                        const int s = s0 + lane;
                        const uint32_t key = s < shi ? keys[s] : kEmpty;
                        const bool occ = key != kEmpty;
                        const unsigned bal = __ballot_sync(SPG_FULL, occ);
                        if (occ) {
                            const int r = o + __popc(bal & ((1u << lane) - 1u));
                            if (r < want) {
                                out_rows[out0 + r] = (I)key;
                                out_vals[out0 + r] = vals[s];
                            }
                        }
                        o += __popc(bal);
                    }
                    if (warp == NW - 1 && lane == 0) sh.pos = o;
                    __syncthreads();
                    if (threadIdx.x == 0) {
                        if (sh.pos != want) atomicOr(c.err, kErrCount);
                        sh.pos = 0;
                    }
                }
                __syncthreads();
            } else {
                // the column's own table in global memory
                const int64_t f = src.flops();   // warp-wide: every warp computes it
                const int64_t rows = f < m ? f : m;
                int log2T = 1;
                while ((1ll << log2T) < 2 * rows) ++log2T;
                const int64_t T = 1ll << log2T;
                uint32_t *keys = mq.gkeys + mq.gtab_off[g];
                V *vals = reinterpret_cast<V *>(mq.gvals) + mq.gtab_off[g];
                for (int64_t s = threadIdx.x; s < T; s += NT) { keys[s] = kEmpty; if (MODE == 1) vals[s] = V(0); }
                __syncthreads();
                int mine = 0;
                auto emit = load_apply(
                    [&](int64_t q, V bv, int64_t) { return RowVal<V>{src.row(q), MODE == 1 ? src.val(q, bv) : V(0)}; },
                    [&](const RowVal<V> &e, bool valid) {
                        if (!valid) return;
                        bool nw;
                        const int64_t h = ghash_insert(keys, log2T, e.r, nw, c.err);
                        if (MODE == 0) mine += nw;
                        else if (h >= 0) gatomic_add_v(&vals[h], e.x);
                    });
                block_walk<kWalkBatch>(src, emit, c.short_seg, c.huge_seg, sh);
                __syncthreads();
                if (MODE == 0) {
                    mine = warp_sum(mine);
                    if (lane == 0) sh.red[warp] = mine;
                    __syncthreads();
                    if (threadIdx.x < 32) {
                        int v = threadIdx.x < NW ? sh.red[threadIdx.x] : 0;
                        v = warp_sum(v);
                        if (threadIdx.x == 0) c.cnt[g] = v;
                    }
                } else {
                    for (int64_t s0 = 0; s0 < T; s0 += NT) {
                        const int64_t s = s0 + threadIdx.x;
                        const uint32_t key = s < T ? keys[s] : kEmpty;
                        const bool occ = key != kEmpty;
                        const unsigned bal = __ballot_sync(SPG_FULL, occ);
                        int wbase = 0;
                        if (lane == 0 && bal) wbase = atomicAdd(&sh.pos, __popc(bal));
                        wbase = __shfl_sync(SPG_FULL, wbase, 0);
                        if (occ) {
                            const int r = wbase + __popc(bal & ((1u << lane) - 1u));
                            if (r < want) {
                                out_rows[out0 + r] = (I)key;
                                out_vals[out0 + r] = vals[s];
                            }
                        }
                    }
                    __syncthreads();
                    if (threadIdx.x == 0) {
                        if (sh.pos != want) atomicOr(c.err, kErrCount);
                        sh.pos = 0;
                    }
                }
                __syncthreads();
            }
        }
    }
    // warp-sized columns: every warp takes kWarpGrab at a time (one counter
    // update per grab), each with a warp-private table, cleared once; a
    // column's output leaves it clean. The walk is the one of k_light.
    constexpr int kWarpGrab = 8;
    V *vals = MODE == 1 ? reinterpret_cast<V *>(smem) + warp * TW : nullptr;
    uint32_t *keys = reinterpret_cast<uint32_t *>(smem + (MODE == 1 ? sizeof(V) * NW * TW : 0)) + warp * TW;
    const unsigned below = (1u << lane) - 1u;
    for (int s = lane; s < TW; s += 32) {
        keys[s] = kEmpty;
        if (MODE == 1) vals[s] = V(0);
    }
    __syncwarp();
    for (;;) {
        long long wb = 0;
        if (lane == 0) wb = (long long)atomicAdd(mq.counter + 1, (unsigned long long)kWarpGrab);
        wb = __shfl_sync(SPG_FULL, wb, 0);
        if (wb >= nwarp) break;
        // the grab's columns, one per lane: column, problem and B range are on
        // their way before the first one is walked
        int64_t gl = 0, b0l = 0;
        int nbl = 0, prl = 0;
        if (lane < kWarpGrab && wb + lane < nwarp) {
            gl = mq.list[mq.off[1] + (int)wb + lane];
            prl = sa.prob_of[gl];
            const auto *p = sa.probs + prl;
            const int64_t bc = gl - p->gcol0;
            b0l = (int64_t)__ldg(&p->bp[bc]);
            nbl = (int)((int64_t)__ldg(&p->bp[bc + 1]) - b0l);
        }
        for (int wi = 0; wi < kWarpGrab && wb + wi < nwarp; ++wi) {
            const int pos = mq.off[1] + (int)wb + wi;
            const int64_t g = __shfl_sync(SPG_FULL, gl, wi);
            const int64_t b0 = __shfl_sync(SPG_FULL, b0l, wi);
            const int nb = __shfl_sync(SPG_FULL, nbl, wi);
            const auto *p = sa.probs + __shfl_sync(SPG_FULL, prl, wi);
            // 2 * cap(t) slots by the column's tier; the numeric pass knows the
            // exact count, usually a smaller table
            int t = 1;
            while (t < wt && mq.off[t + 1] <= pos) ++t;
            int64_t out0 = 0;
            int want = tier_cap(t);
            if (MODE == 1) {
                out0 = c.colptr[g] - c.out_base;
                want = (int)min(c.colptr[g + 1] - c.colptr[g], (int64_t)want);
            }
            int log2T = 6;
            while ((1 << log2T) < 2 * want) ++log2T;
            const int T = 1 << log2T;
            int mine = 0;
            auto insert = [&](uint32_t r, V x) {
                bool nw;
                const int h = hash_insert_dbl1(keys, log2T, r, c.err, nw);
                if (MODE == 0) mine += nw;
                else if (h >= 0) atomic_add_v(&vals[h], x);
            };
            walk_entries<MODE>(p, 0, INT64_MAX, b0, nb, 0, 1, 0, 1, s_off[warp], s_bv[MODE == 1 ? warp : 0], insert);
            if (MODE == 0) {
                mine = warp_sum(mine);
                if (lane == 0) c.cnt[g] = mine;
                uint4 *k4 = reinterpret_cast<uint4 *>(keys);
                for (int s = lane; s < T / 4; s += 32) k4[s] = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
            } else {
                int pos2 = 0;
                for (int s0 = 0; s0 < T; s0 += 32) {
                    const int s = s0 + lane;
                    const uint32_t key = keys[s];
                    const bool occ = key != kEmpty;
                    const unsigned bal = __ballot_sync(SPG_FULL, occ);
                    if (occ) {
                        const int r = pos2 + __popc(bal & below);
                        if (r < want) {
                            out_rows[out0 + r] = (I)key;
                            out_vals[out0 + r] = vals[s];
                        }
                        keys[s] = kEmpty;
                        vals[s] = V(0);
                    }
                    pos2 += __popc(bal);
                }
                if (lane == 0 && pos2 != want) atomicOr(c.err, kErrCount);
            }
            __syncwarp();
        }
    }
}

// Table sizes of the heavy columns of the multi-problem product (2 * min(f_j,
// m) slots rounded up to a power of two; 0 for the other columns); their
// exclusive scan places each column's global table.
template <class Src>
__global__ void k_multi_gtab_sizes(typename Src::Args sa, const int64_t *f, const uint8_t *tier, int64_t n,
                                   int64_t *size) {
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n) return;
    int64_t sz = 0;
    if (tier[g] >= kHeavyTier0) {
        Src src;
        src.open(sa, g);
        const int64_t m = src.m();
        const int64_t rows = f[g] < m ? f[g] : m;
        sz = 2;
        while (sz < 2 * rows) sz <<= 1;
    }
    size[g] = sz;
}

}  // namespace spg
