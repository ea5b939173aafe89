// Non-templated helper kernels: numeric tiering, tier scatter, int64 scans,
// small copies.
#include "util.h"
#include "kernels.cuh"

namespace spg {

__global__ void k_numeric_tier(const int64_t *cnt, const int64_t *dense_sel, int64_t c_lo,
                               int64_t c_hi, int hash_cap_max, uint8_t *tier_out,
                               int32_t *tier_hist) {
    __shared__ int s_hist[kTiers];
    if (threadIdx.x < kTiers) s_hist[threadIdx.x] = 0;
    __syncthreads();
    const int64_t g = c_lo + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g < c_hi) {
        const int t = num_tier(cnt[g], dense_sel ? dense_sel[g] : 0, hash_cap_max);
        tier_out[g] = (uint8_t)t;
        if (t) atomicAdd(&s_hist[t], 1);
    }
    __syncthreads();
    if (threadIdx.x < kTiers && s_hist[threadIdx.x]) atomicAdd(&tier_hist[threadIdx.x], s_hist[threadIdx.x]);
}

__global__ void __launch_bounds__(kTierBlock) k_tier_blocks(const int64_t *cp, const int64_t *sel, int64_t n,
                                                             int hash_cap_max, int32_t *blk, const int *err,
                                                             int32_t *err_out) {
    __shared__ int s_hist[kTiers];
    if (threadIdx.x < kTiers) s_hist[threadIdx.x] = 0;
    __syncthreads();
    const int64_t g = (int64_t)blockIdx.x * kTierBlock + threadIdx.x;
    if (g < n)
        atomicAdd(&s_hist[num_tier(cp[g + 1] - cp[g], sel ? sel[g + 1] - sel[g] : 0, hash_cap_max)], 1);
    __syncthreads();
    if (threadIdx.x < kTiers && n > 0) blk[(int64_t)blockIdx.x * 16 + threadIdx.x] = s_hist[threadIdx.x];
    if (blockIdx.x == 0 && threadIdx.x == 0) *err_out = *err;
}

__global__ void k_bin_scatter(const uint8_t *tier, int64_t c_lo, int64_t c_hi,
                              const int32_t *tier_hist, int32_t *cursor, int32_t *list,
                              int32_t *list_off, int32_t *heavy_ord) {
    __shared__ int s_off[kTiers + 1];
    __shared__ int s_cnt[kTiers];
    __shared__ int s_base[kTiers];
    if (threadIdx.x == 0) {
        int acc = 0;
        for (int t = 0; t < kTiers; ++t) { s_off[t] = acc; acc += (t == 0 ? 0 : tier_hist[t]); }
        s_off[kTiers] = acc;
        if (blockIdx.x == 0)
            for (int t = 0; t <= kTiers; ++t) list_off[t] = s_off[t];
    }
    if (threadIdx.x < kTiers) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    const int64_t g = c_lo + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int t = 0, rank = 0;
    if (g < c_hi) {
        t = tier[g];
        if (t) rank = atomicAdd(&s_cnt[t], 1);
    }
    __syncthreads();
    if (threadIdx.x < kTiers && s_cnt[threadIdx.x])
        s_base[threadIdx.x] = atomicAdd(&cursor[threadIdx.x], s_cnt[threadIdx.x]);
    __syncthreads();
    if (g < c_hi && t) {
        const int pos = s_off[t] + s_base[t] + rank;
        list[pos] = (int32_t)g;
        if (heavy_ord && t >= kHeavyTier0) heavy_ord[g] = pos - s_off[kHeavyTier0];
    }
}

// One CTA for up to kBinSmall columns, a run of them per warp and step: lanes of
// one tier take their places with one shared add. It replaces a memset, the tier
// kernel and the scatter: a 64 x 64 product has 11 launches and copies with
// it, one memset for the symbolic step's words and one copy back, 17 without
// (step 240 -> 222 us; a uniform 4096-column product 254 -> 236 us).
__global__ void __launch_bounds__(1024) k_bin_small(const int64_t *f, int64_t m, int cap_full, const int64_t *num_cnt,
                                                    const int64_t *num_sel, int64_t c_lo, int n, int hash_cap_max,
                                                    uint8_t *tier, int64_t *cnt_out, int32_t *list, int32_t *list_off,
                                                    int32_t *heavy_ord, int32_t *hist, int32_t *over,
                                                    int32_t *cursor) {
    __shared__ int s_cnt[kTiers], s_off[kTiers + 1], s_over;
    __shared__ unsigned long long s_above[3];
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < kTiers) s_cnt[threadIdx.x] = 0;
    if (threadIdx.x == 0) s_over = 0;
    if (threadIdx.x < 3) s_above[threadIdx.x] = 0;
    if (threadIdx.x < 64) cursor[threadIdx.x] = 0;
    __syncthreads();
    constexpr int kPer = kBinSmall / 1024;
    int mine[kPer];   // tier and rank inside the tier
    const bool rule = f && hash_cap_max < cap_full;
    AboveSums above;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        mine[i] = 0;
        const int j = i * 1024 + (int)threadIdx.x;
        if (i * 1024 >= n) break;   // the same for the CTA
        int t = 0;
        if (j < n) {
            const int64_t g = c_lo + j;
            if (f) {
                const int64_t u = f[g] < m ? f[g] : m;
                if (u > cap_full) atomicAdd(&s_over, 1);
                if (rule && u > hash_cap_max) above.add(f[g]);
                t = hash_tier_of(u, hash_cap_max);
                if (t < 0) t = heavy_subtier(u);
                cnt_out[g] = 0;
            } else {
                t = num_tier(num_cnt[g], num_sel ? num_sel[g] : 0, hash_cap_max);
            }
            tier[g] = (uint8_t)t;
        }
        const unsigned peers = __match_any_sync(SPG_FULL, t);
        const int lead = __ffs(peers) - 1;
        int base = 0;
        if (t && lane == lead) base = atomicAdd(&s_cnt[t], __popc(peers));
        base = __shfl_sync(SPG_FULL, base, lead);
        mine[i] = t | (base + __popc(peers & ((1u << lane) - 1u))) << 5;
    }
    if (rule) above.warp_add(s_above);
    __syncthreads();
    if (threadIdx.x == 0) {
        int acc = 0;
        for (int t = 0; t < kTiers; ++t) { s_off[t] = acc; acc += t ? s_cnt[t] : 0; }
        s_off[kTiers] = acc;
        if (over) {
            *over = s_over;
            for (int i = 0; i < 3; ++i) reinterpret_cast<unsigned long long *>(over + 2)[i] = s_above[i];
        }
    }
    __syncthreads();
    if (threadIdx.x <= kTiers) list_off[threadIdx.x] = s_off[threadIdx.x];
    if (threadIdx.x < kTiers) hist[threadIdx.x] = s_cnt[threadIdx.x];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int j = i * 1024 + (int)threadIdx.x;
        const int t = mine[i] & 31;
        if (j < n && t) {
            const int pos = s_off[t] + (mine[i] >> 5);
            list[pos] = (int32_t)(c_lo + j);
            if (heavy_ord && t >= kHeavyTier0) heavy_ord[c_lo + j] = pos - s_off[kHeavyTier0];
        }
    }
}

// Cuts heavy column h (global column g) into its items, in panel order:
// emit(kind, HeavyItem) with kind 0 for dense and 1 for hash items.
template <class F>
__device__ __forceinline__ void cut_items(int64_t g, const int32_t *pc, int P, int dense_min, int range_cap,
                                          int max_panels, F &&emit) {
    int gp0 = -1, gcnt = 0, off = 0, goff = 0;
    auto flush = [&](int p_end) {
        if (gp0 >= 0 && gcnt > 0) emit(1, HeavyItem{(int32_t)g, gp0, p_end, gcnt, goff, 0});
        gp0 = -1; gcnt = 0;
    };
    for (int p = 0; p < P; ++p) {
        const int x = pc[p];
        if (x >= dense_min) {
            flush(p);
            emit(0, HeavyItem{(int32_t)g, p, p + 1, -x, off, 0});
            off += x;
            continue;
        }
        if (gp0 >= 0 && (gcnt + x > range_cap || p - gp0 >= max_panels)) flush(p);
        if (x == 0 && gp0 < 0) continue;      // no open group: skip empty panels
        if (gp0 < 0) { gp0 = p; goff = off; }
        gcnt += x;
        off += x;
    }
    flush(P);
}

// mode 0: bins[kind * P + first panel] += items; mode 1: bins hold the bins'
// first positions, every item is written at the next position of its bin
// (dense items before hash items, each by first panel). One thread per heavy
// column runs the greedy cut over its P panel counts. For up to kItemBins bins
// a CTA counts its items in shared memory and takes each bin's run with one
// global atomic. Mode 0 also adds the items of columns above cap_full to
// bins[2 P].
__global__ void __launch_bounds__(256) k_heavy_items(const int32_t *list, const int32_t *list_off, const int64_t *sel,
                                                     int hash_cap_max, int cap_full, const int32_t *pcnt, int P, int dense_min,
                                                     int range_cap, int max_panels, int mode, int32_t *bins,
                                                     HeavyItem *items, int32_t *order) {
    __shared__ int s_cnt[kItemBins], s_base[kItemBins];
    const int lo = list_off[kHeavyTier0], hi = list_off[kTiers];
    const int64_t h = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int nbins = 2 * P;
    const bool local = nbins <= kItemBins;
    const int64_t g = h < hi - lo ? list[lo + h] : 0;
    const bool mine = h < hi - lo && sel[g] > hash_cap_max;
    const int32_t *pc = pcnt + h * P;
    if (mode == 0) {
        int full = 0;
        if (mine && sel[g] > cap_full)
            cut_items(g, pc, P, dense_min, range_cap, max_panels, [&](int, const HeavyItem &) { ++full; });
        full = warp_sum(full);
        if ((threadIdx.x & 31) == 0 && full) atomicAdd(&bins[nbins], full);
    }
    if (local) {
        for (int b = threadIdx.x; b < nbins; b += blockDim.x) s_cnt[b] = 0;
        __syncthreads();
        if (mine)
            cut_items(g, pc, P, dense_min, range_cap, max_panels,
                      [&](int kind, const HeavyItem &it) { atomicAdd(&s_cnt[kind * P + it.p0], 1); });
        __syncthreads();
        for (int b = threadIdx.x; b < nbins; b += blockDim.x) {
            s_base[b] = s_cnt[b] ? atomicAdd(&bins[b], s_cnt[b]) : 0;
            s_cnt[b] = 0;
        }
        if (mode == 0) return;
        __syncthreads();
    }
    if (mine)
        cut_items(g, pc, P, dense_min, range_cap, max_panels, [&](int kind, const HeavyItem &it) {
            const int b = kind * P + it.p0;
            const int at = local ? s_base[b] + atomicAdd(&s_cnt[b], 1) : atomicAdd(&bins[b], 1);
            if (mode) { items[at] = it; order[at] = at; }
        });
}

// The same in one launch of one CTA, for few columns and panels (nheavy * P
// <= kItemsOne): counts, bin prefix, items if there is room for them, and the
// totals (of all items, of those of columns above cap_full).
__global__ void __launch_bounds__(1024) k_heavy_items_one(const int32_t *list, const int32_t *list_off,
                                                          const int64_t *sel, int hash_cap_max, int cap_full,
                                                          const int32_t *pcnt, int P, int dense_min, int range_cap, int max_panels,
                                                          int64_t room, HeavyItem *items, int32_t *order,
                                                          int64_t *total) {
    __shared__ int s_bin[kItemBins];
    __shared__ int s_full;
    if (threadIdx.x == 0) s_full = 0;
    const int lo = list_off[kHeavyTier0], nh = list_off[kTiers] - lo;
    const int nbins = 2 * P;
    for (int b = threadIdx.x; b < nbins; b += blockDim.x) s_bin[b] = 0;
    __syncthreads();
    for (int h = threadIdx.x; h < nh; h += blockDim.x) {
        const int64_t g = list[lo + h];
        if (sel[g] > hash_cap_max)
            cut_items(g, pcnt + (int64_t)h * P, P, dense_min, range_cap, max_panels,
                      [&](int kind, const HeavyItem &it) {
                          atomicAdd(&s_bin[kind * P + it.p0], 1);
                          if (sel[g] > cap_full) atomicAdd(&s_full, 1);
                      });
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        int carry = 0;
        for (int b0 = 0; b0 < nbins; b0 += 32) {
            const int b = b0 + threadIdx.x;
            const int v = b < nbins ? s_bin[b] : 0;
            const int incl = warp_incl_scan(v);
            if (b < nbins) s_bin[b] = carry + incl - v;
            carry += __shfl_sync(SPG_FULL, incl, 31);
        }
        if (threadIdx.x == 0) { total[0] = carry; total[1] = s_full; }
    }
    __syncthreads();
    for (int h = threadIdx.x; h < nh; h += blockDim.x) {
        const int64_t g = list[lo + h];
        if (sel[g] > hash_cap_max)
            cut_items(g, pcnt + (int64_t)h * P, P, dense_min, range_cap, max_panels,
                      [&](int kind, const HeavyItem &it) {
                          const int at = atomicAdd(&s_bin[kind * P + it.p0], 1);
                          if (at < room) { items[at] = it; order[at] = at; }
                      });
    }
}

__global__ void k_panel_starts(int64_t ka, int P, int32_t *apo, int64_t *ape) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < ka;
         k += (int64_t)gridDim.x * blockDim.x) {
        int32_t *o = apo + k * ((int64_t)P + 1) + 1;
        int32_t run = 0;
#pragma unroll 4
        for (int p = 0; p < P; ++p) {
            const int32_t c = o[p];
            ape[(int64_t)p * ka + k] = c;
            o[p] = run;
            run += c;
        }
    }
}

__global__ void k_items_by_batch(const HeavyItem *items, int64_t n, const int64_t *bounds, int64_t nb,
                                 int pe, int mode, unsigned long long *cnt, int32_t *order) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const HeavyItem it = items[i];
        const int64_t g = it.g;
        // the batch t with bounds[t] <= g < bounds[t + 1]
        int64_t lo = 0, hi = nb - 1;
        while (lo < hi) {
            const int64_t mid = (lo + hi + 1) >> 1;
            if (bounds[mid] <= g) lo = mid; else hi = mid - 1;
        }
        // dense items (cnt < 0) before hash items inside a batch
        const int64_t key = (lo * 2 + (it.cnt < 0 ? 0 : 1)) * pe + (pe > 1 ? it.p0 : 0);
        if (mode == 0) atomicAdd(&cnt[key], 1ull);
        else order[atomicAdd(&cnt[key], 1ull)] = (int32_t)i;
    }
}

// After the scatter cnt[key] is the end of bucket key; a batch has 2 * pe
// buckets, so batch t starts at cnt[t * 2 * pe - 1] (0 for t = 0) and
// start[nb] = n.
__global__ void k_batch_item_starts(const unsigned long long *cnt, int64_t nb, int pe, int64_t n,
                                    int64_t *start) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t > nb) return;
    start[t] = t == 0 ? 0 : t == nb ? n : (int64_t)cnt[t * 2 * pe - 1];
}

// exclusive scan of n ints in place (one CTA); the sum goes to total[0], a[n] to
// total[1]
__global__ void __launch_bounds__(1024) k_small_excl_scan(int32_t *a, int n, int64_t *total) {
    __shared__ int32_t s_warp[33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t carry = 0;
    for (int base = 0; base < n; base += 1024) {
        const int i = base + threadIdx.x;
        const int32_t v = i < n ? a[i] : 0;
        const int32_t incl = warp_incl_scan(v);
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        const int32_t w = s_warp[lane];
        const int32_t wi = warp_incl_scan(w);
        const int32_t before = __shfl_sync(SPG_FULL, wi - w, warp);
        const int32_t all = __shfl_sync(SPG_FULL, wi, 31);
        if (i < n) a[i] = carry + before + incl - v;
        carry += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) { total[0] = carry; total[1] = a[n]; }
}

// ---- exclusive scan of int64 (three phases, all on the device) ------------
constexpr int kScanThreads = 1024;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ int64_t block_excl_scan(int64_t v, int64_t *s_warp, int64_t &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t incl = warp_incl_scan(v);
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int64_t w = lane < (int)(blockDim.x >> 5) ? s_warp[lane] : 0;
        int64_t wi = warp_incl_scan(w);
        s_warp[lane] = wi - w;
        if (lane == 31) s_warp[32] = wi;
    }
    __syncthreads();
    int64_t r = s_warp[warp] + incl - v;
    total = s_warp[32];
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(const int64_t *in, int64_t n,
                                                              int64_t *partials) {
    __shared__ int64_t s_warp[33];
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    int64_t s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        const int64_t idx = base + (int64_t)i * kScanThreads + threadIdx.x;
        if (idx < n) s += in[idx];
    }
    int64_t total;
    block_excl_scan(s, s_warp, total);
    if (threadIdx.x == 0) partials[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_partials(int64_t *partials, int64_t np) {
    __shared__ int64_t s_warp[33];
    int64_t carry = 0;
    for (int64_t b = 0; b < np; b += kScanThreads) {
        const int64_t i = b + threadIdx.x;
        int64_t v = i < np ? partials[i] : 0;
        int64_t total;
        int64_t ex = block_excl_scan(v, s_warp, total);
        if (i < np) partials[i] = ex + carry;
        carry += total;
    }
    if (threadIdx.x == 0) partials[np] = carry;
}

// A CTA's exclusive scan of the ITEMS * kScanThreads entries at t0, plus
// `before`. A warp owns a run of 32 * ITEMS entries in rows of 32, so every load and
// store is a full line; returns the tile's total.
template <int ITEMS>
__device__ __forceinline__ int64_t scan_tile(const int64_t *in, int64_t n, int64_t t0, int64_t before, int64_t *out,
                                             int64_t *s_warp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t base = t0 + (int64_t)warp * (32 * ITEMS) + lane;
    int64_t v[ITEMS], ex[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) v[i] = base + 32 * i < n ? in[base + 32 * i] : 0;
    int64_t run = 0;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const int64_t incl = warp_incl_scan(v[i]);
        ex[i] = run + incl - v[i];
        run += __shfl_sync(SPG_FULL, incl, 31);
    }
    int64_t total;
    if (lane == 0) s_warp[warp] = run;
    __syncthreads();
    const int64_t w = s_warp[lane];   // kScanThreads / 32 == 32 warps
    const int64_t wi = warp_incl_scan(w);
    before += __shfl_sync(SPG_FULL, wi - w, warp);
    total = __shfl_sync(SPG_FULL, wi, 31);
#pragma unroll
    for (int i = 0; i < ITEMS; ++i)
        if (base + 32 * i < n) out[base + 32 * i] = before + ex[i];
    return total;
}

// out[i] = sum_{j<i} in[j] for i in [0, n]; in and out may alias. np > 0: the
// partials are the tiles' own sums, and every CTA adds up those before its
// tile (np of them at most); np == 0: they are prefixes already.
__global__ void __launch_bounds__(kScanThreads) k_scan_apply(const int64_t *in, int64_t n,
                                                             const int64_t *partials, int np,
                                                             int64_t *out, int write_total) {
    __shared__ int64_t s_warp[33];
    int64_t before = 0;
    if (np > 0) {
        int64_t p = 0;
        for (int i = threadIdx.x; i < (int)blockIdx.x; i += kScanThreads) p += partials[i];
        block_excl_scan(p, s_warp, before);
    } else if (partials) {
        before = partials[blockIdx.x];
    }
    const int64_t total = scan_tile<kScanItems>(in, n, (int64_t)blockIdx.x * kScanTile, before, out, s_warp);
    if (write_total && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[n] = before + total;
}

// The whole scan in one launch, for in != out and small n: every CTA first
// sums all the input before its tile (from L2), then scans its tile.
constexpr int kDirectItems = 2;
constexpr int kDirectTile = kDirectItems * kScanThreads;
__global__ void __launch_bounds__(kScanThreads) k_scan_direct(const int64_t *in, int64_t n, int64_t *out,
                                                              int write_total) {
    __shared__ int64_t s_warp[33];
    const int64_t t0 = (int64_t)blockIdx.x * kDirectTile;
    int64_t p = 0, before;
#pragma unroll 16
    for (int64_t i = threadIdx.x; i < t0; i += kScanThreads) p += in[i];
    block_excl_scan(p, s_warp, before);
    const int64_t total = scan_tile<kDirectItems>(in, n, t0, before, out, s_warp);
    if (write_total && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[n] = before + total;
}

int64_t scan_partials_len(int64_t n) { return (n + kScanTile - 1) / kScanTile + 1; }

// The form by size. One launch up to kDirectScan entries: a CTA reads on
// average half the input again, which costs less than a second launch (50,021 entries: 7.5 us
// against 2.7 + 6.0 us and a launch; even at 65,536: 10.0 against 8.8 us).
// Up to kFoldPartials tiles the apply kernel adds up the partials itself,
// which saves the launch between (3 us). Beyond, three launches.
constexpr int64_t kDirectScan = 56 * 1024;
constexpr int64_t kFoldPartials = 1024;
int scan_launches(int64_t n, bool in_place) {
    const int64_t nb = n > 0 ? (n + kScanTile - 1) / kScanTile : 1;
    if ((!in_place && n <= kDirectScan) || nb == 1) return 1;
    return nb <= kFoldPartials ? 2 : 3;
}
cudaError_t exclusive_scan_i64(const int64_t *in, int64_t n, int64_t *out, int64_t *partials,
                               int write_total, cudaStream_t st) {
    const int64_t nb = n > 0 ? (n + kScanTile - 1) / kScanTile : 1;
    if (in != out && n <= kDirectScan) {
        const int64_t nd = n > 0 ? (n + kDirectTile - 1) / kDirectTile : 1;
        k_scan_direct<<<(unsigned)nd, kScanThreads, 0, st>>>(in, n, out, write_total);
    } else if (nb == 1) {
        k_scan_apply<<<1, kScanThreads, 0, st>>>(in, n, nullptr, 0, out, write_total);
    } else {
        k_scan_reduce<<<(unsigned)nb, kScanThreads, 0, st>>>(in, n, partials);
        const bool fold = nb <= kFoldPartials;
        if (!fold) k_scan_partials<<<1, kScanThreads, 0, st>>>(partials, nb);
        k_scan_apply<<<(unsigned)nb, kScanThreads, 0, st>>>(in, n, partials, fold ? (int)nb : 0, out, write_total);
    }
    return cudaGetLastError();
}

// ---- small kernels ----------------------------------------------------------

// dst[i] = src[i] - src[0] for i in [0, n], narrowed to the output pointer type.
__global__ void k_rebase_colptr_i64(const int64_t *src, int64_t n, int64_t *dst) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i <= n) dst[i] = src[i] - src[0];
}
__global__ void k_rebase_colptr_i32(const int64_t *src, int64_t n, int32_t *dst) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i <= n) dst[i] = (int32_t)(src[i] - src[0]);
}

cudaError_t rebase_colptr(const int64_t *src, int64_t n, void *dst, int dst_is_i64,
                          cudaStream_t st) {
    const unsigned nb = (unsigned)((n + 1 + 255) / 256);
    if (dst_is_i64) k_rebase_colptr_i64<<<nb, 256, 0, st>>>(src, n, (int64_t *)dst);
    else k_rebase_colptr_i32<<<nb, 256, 0, st>>>(src, n, (int32_t *)dst);
    return cudaGetLastError();
}

// Validation of a CSC: colptr monotone from 0 to nnz, rows in [0, nrows).
template <class I>
__global__ void k_validate(const I *colptr, const I *rowidx, int64_t ncols, int64_t nrows,
                           int64_t nnz, int *bad) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i <= ncols; i += stride) {
        const int64_t c = (int64_t)colptr[i];
        if (i == 0 && c != 0) atomicOr(bad, 1);
        if (i == ncols && c != nnz) atomicOr(bad, 1);
        if (i < ncols && (int64_t)colptr[i + 1] < c) atomicOr(bad, 1);
    }
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nnz; i += stride) {
        const int64_t r = (int64_t)rowidx[i];
        if (r < 0 || r >= nrows) atomicOr(bad, 2);
    }
}

cudaError_t validate_csc(const void *colptr, const void *rowidx, int idx64, int64_t ncols,
                         int64_t nrows, int64_t nnz, int *d_bad, cudaStream_t st) {
    const unsigned nb = 1024;
    if (idx64)
        k_validate<int64_t><<<nb, 256, 0, st>>>((const int64_t *)colptr, (const int64_t *)rowidx,
                                                ncols, nrows, nnz, d_bad);
    else
        k_validate<int32_t><<<nb, 256, 0, st>>>((const int32_t *)colptr, (const int32_t *)rowidx,
                                                ncols, nrows, nnz, d_bad);
    return cudaGetLastError();
}

// w[g] = bytes_per_nnz * (cnt[g] + extra[g]) + ptr_bytes, for g in [0, n).
__global__ void k_column_bytes(const int64_t *cnt, const int64_t *extra, int64_t n, int64_t r,
                               int64_t ptr_bytes, int64_t *w) {
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g < n) w[g] = r * (cnt[g] + (extra ? extra[g] : 0)) + ptr_bytes;
}

cudaError_t column_bytes(const int64_t *cnt, const int64_t *extra, int64_t n, int64_t r,
                         int64_t ptr_bytes, int64_t *w, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    k_column_bytes<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(cnt, extra, n, r, ptr_bytes, w);
    return cudaGetLastError();
}

__global__ void k_add_i64(int64_t *dst, const int64_t *src, int64_t n) {
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g < n) dst[g] += src[g];
}

cudaError_t add_i64(int64_t *dst, const int64_t *src, int64_t n, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    k_add_i64<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(dst, src, n);
    return cudaGetLastError();
}

}  // namespace spg
