// Typed host driver of the kernels: symbolic step, batch plan, numeric step
// (plain or k-split + hash merge), standalone merge, backward.
#pragma once

#include <algorithm>
#include <array>
#include <cmath>
#include <cstring>
#include <functional>
#include <type_traits>
#include <vector>

#include "kernels.cuh"
#include "sort_prune.cuh"
#include "plan.h"
#include "util.h"

namespace spg {

#define SPG_CK(call)                                                   \
    do {                                                               \
        cudaError_t e_ = (call);                                       \
        if (e_ != cudaSuccess) return cuda_fail(e_, #call);            \
    } while (0)

#define SPG_ST(...)                                                    \
    do {                                                               \
        spgemm_status s_ = (__VA_ARGS__);                              \
        if (s_ != SPGEMM_OK) return s_;                                \
    } while (0)

inline int block_tier_threads(int T, const Tuning &tun) {
    if (tun.block_threads) return tun.block_threads;
    if (T <= 1024) return 128;
    if (T <= 4096) return 256;
    if (T <= 8192) return 512;
    return 1024;
}

// The binning words of a pass, zeroed together: [0, 16) tier histogram,
// [kFlopTotal, +2) total multiplications (64 bits), [kOverFull] columns above
// the plan's largest hash table, [kAbove, +6) sums over the columns above the line in
// use (three of 64 bits, see k_col_tier), [64, 128) list cursors and the work counters of
// the persistent kernels.
constexpr int kBinInts = 128;
constexpr int kFlopTotal = 32;
constexpr int kOverFull = 34;
constexpr int kAbove = kOverFull + 2;

// Scratch shared by one symbolic / numeric pass.
struct Ctx {
    int nsm;
    Tuning tun;
    int *err;
    int32_t *hist;       // kBinInts ints: tier histogram, flop total, cursors
    int32_t *cursor;     // hist + 64: list cursors, work counters
    int32_t *h_small;    // pinned host, >= 64 ints
    int P, Q;
    int64_t Rs;
    PhaseTimer *tm = nullptr;   // optional phase timing and launch counting
    int ph_hash = kPhNumHash, ph_dense = kPhNumDense;
    bool stage_items = false;   // heavy items take their counts from pcnt_in
    int cap_full = 8192;        // the plan's largest hash table
    int over_full = 0;          // sym_pass: columns that may exceed it
    bool sort = false;          // the pass writes C itself in row order (opts.sort_output)
    const int64_t *f = nullptr; // flops per column of the full product (hybrid accumulator)
    int tbegin(int phase, cudaStream_t st) const { return tm ? tm->begin(phase, st) : -1; }
    void tend(int idx, cudaStream_t st) const { if (tm) tm->end(idx, st); }
    void launched(int n = 1) const { if (tm) tm->launches += n; }
};

inline Ctx make_ctx(PlanState &ps) {
    Ctx c;
    c.tm = &ps.timer;
    c.nsm = ps.nsm; c.tun = ps.tun; c.err = ps.err.as<int>();
    c.hist = ps.hist.as<int32_t>(); c.cursor = c.hist + 64;
    c.h_small = ps.h_small.as<int32_t>();
    c.P = ps.P; c.Q = ps.Q; c.Rs = ps.Rs;
    c.f = ps.f.as<int64_t>();
    c.cap_full = ps.cap_full;
    return c;
}

inline TierCommon common_of(const Ctx &c) {
    TierCommon t{};
    t.short_seg = c.tun.short_seg;
    t.huge_seg = c.tun.huge_seg;
    t.err = c.err;
    t.hash_cap_max = c.tun.hash_cap_max;
    t.P = c.P; t.log2R = c.tun.log2R; t.Rs = c.Rs; t.Q = c.Q;
    t.flops = c.f;
    t.hybrid_sort = c.tun.hybrid_sort;
    t.sort = c.sort ? 1 : 0;
    return t;
}

// Allow a kernel the largest dynamic shared memory the device permits next to
// its static shared memory (opt-in maximum minus static size).
template <class K> static void set_smem(K kern) {
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, kern) == cudaSuccess && optin > (int)fa.sharedSizeBytes)
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             optin - (int)fa.sharedSizeBytes);
    cudaGetLastError();   // attribute calls must not leave a sticky error behind
}

// Output of a numeric pass.
template <class I, class V> struct NumOut {
    const int64_t *colptr;
    int64_t out_base;
    I *rows;
    V *vals;
};

// The columns above the hash line: their number, and k_col_tier's sums of their
// multiplications, of the logarithms (in 64ths) and of the squares of these.
struct Above {
    int64_t n = 0, sum = 0, lg = 0, sq = 0;
};

template <class I, class V> struct Engine : EngineBase {
    using PD = ProbDev<I, V>;
    using GA = GemmArgs<I, V>;
    using PA = PartsArgs<I, V>;

    // ---- function attributes ------------------------------------------------
    // the shared memory limits of the kernels, which belong to a context
    static void attrs() {
        static ContextOnce once;
        once.run([] { set_limits(); });
    }
    static void set_limits() {
        set_smem(k_sym_block<SrcGemm<I, V>, 512>);
        set_smem(k_sym_block<SrcGemm<I, V>, 1024>);
        set_smem(k_sym_block<SrcGemm<I, V>, 2048>);
        set_smem(k_sym_block<SrcGemm<I, V>, 4096>);
        set_smem(k_sym_block<SrcGemm<I, V>, 8192>);
        set_smem(k_sym_block<SrcGemm<I, V>, 16384>);
        set_smem(k_sym_block<SrcParts<I, V>, 512>);
        set_smem(k_sym_block<SrcParts<I, V>, 1024>);
        set_smem(k_sym_block<SrcParts<I, V>, 2048>);
        set_smem(k_sym_block<SrcParts<I, V>, 4096>);
        set_smem(k_sym_block<SrcParts<I, V>, 8192>);
        set_smem(k_sym_block<SrcParts<I, V>, 16384>);
        set_smem(k_num_block<SrcGemm<I, V>, 512>);
        set_smem(k_num_block<SrcGemm<I, V>, 1024>);
        set_smem(k_num_block<SrcGemm<I, V>, 2048>);
        set_smem(k_num_block<SrcGemm<I, V>, 4096>);
        set_smem(k_num_block<SrcGemm<I, V>, 8192>);
        set_smem(k_num_block<SrcGemm<I, V>, 16384>);
        set_smem(k_num_block<SrcParts<I, V>, 512>);
        set_smem(k_num_block<SrcParts<I, V>, 1024>);
        set_smem(k_num_block<SrcParts<I, V>, 2048>);
        set_smem(k_num_block<SrcParts<I, V>, 4096>);
        set_smem(k_num_block<SrcParts<I, V>, 8192>);
        set_smem(k_num_block<SrcParts<I, V>, 16384>);
        set_smem(k_bwd_block<I, V, 512>);
        set_smem(k_bwd_block<I, V, 1024>);
        set_smem(k_bwd_block<I, V, 2048>);
        set_smem(k_bwd_block<I, V, 4096>);
        set_smem(k_bwd_block<I, V, 8192>);
        set_smem(k_bwd_block<I, V, 16384>);
        set_smem(k_sym_bitmap<SrcGemm<I, V>>);
        set_smem(k_sym_heavy32<I, V, 1024, 1>);
        set_smem(k_sym_heavy32<I, V, 512, 3>);
        set_smem(k_sym_bitmap<SrcParts<I, V>>);
        set_smem(k_num_dense<SrcPanel<I, V>>);
        set_smem(k_num_dense<SrcPartsPanel<I, V>>);
        set_smem(k_bwd_dense<I, V>);
        set_smem(k_mid<I, V, 4096, 0>);
        set_smem(k_mid<I, V, 4096, 1>);
        set_smem(k_mid<I, V, 8192, 0>);
        set_smem(k_mid<I, V, 8192, 1>);
        set_smem(k_mid<I, V, 16384, 0>);
        set_smem(k_mid<I, V, 16384, 1>);
        set_smem(k_light<I, V, 1024, 0>);
        set_smem(k_light<I, V, 512, 1>);
        set_smem(k_light<I, V, 1024, 1>);
        set_smem(k_sym_warp<SrcGemm<I, V>, 1024>);
        set_smem(k_sym_warp<SrcParts<I, V>, 1024>);
        set_smem(k_num_warp<SrcGemm<I, V>, 512>);
        set_smem(k_num_warp<SrcGemm<I, V>, 1024>);
        set_smem(k_num_warp<SrcParts<I, V>, 512>);
        set_smem(k_num_warp<SrcParts<I, V>, 1024>);
        set_smem(k_bwd_light<I, V, 512>);
        set_smem(k_bwd_light<I, V, 1024>);
        set_smem(k_bwd_warp<I, V, 512>);
        set_smem(k_bwd_warp<I, V, 1024>);
        set_smem(k_num_heavy<SrcPanelRange<I, V>, SrcColRange<I, V>, 2>);
        set_smem(k_num_heavy<SrcPartsRange<I, V>, SrcPartsRange<I, V>, 2>);
        set_smem(k_num_heavy<SrcPanelRange<I, V>, SrcColRange<I, V>, 3>);
        set_smem(k_num_heavy<SrcPartsRange<I, V>, SrcPartsRange<I, V>, 3>);
        set_smem(k_multi_pass<SrcGemm<I, V>, 512, 0>);
        set_smem(k_multi_pass<SrcGemm<I, V>, 512, 1>);
        set_smem(k_multi_pass<SrcGemm<I, V>, 256, 0>);
        set_smem(k_multi_pass<SrcGemm<I, V>, 256, 1>);
        set_smem(k_multi_pass<SrcGemm<I, V>, 128, 0>);
        set_smem(k_multi_pass<SrcGemm<I, V>, 128, 1>);
        set_smem(k_num_heavy32<I, V, 1, false>);
        set_smem(k_num_heavy32<I, V, 1, true>);
        set_smem(k_num_heavy32<I, V, 2, false>);
        set_smem(k_num_heavy32<I, V, 2, true>);
        set_smem(k_num_heavy32<I, V, 3, false>);
        set_smem(k_num_heavy32<I, V, 3, true>);
        set_smem(k_sort_cols<I, V, 512, false>);
        set_smem(k_sort_cols<I, V, 2048, true>);
        set_smem(k_sort_cols<I, V, 16384, true>);
        set_smem(k_prune_select<I, V, I>);
        set_smem(k_sort_items<I, V, 8192>);
        set_smem(k_sort_items<I, V, 4096>);
    }

    // ---- tier launches -----------------------------------------------------
    // A CTA tier of a product with 32-bit stream positions (narrow; larger products
    // keep block_walk). count < 0: population unknown.
    static bool launch_mid(const Ctx &cx, const GA &sa, const TierCommon &c, int T, int thr, int mode, int count,
                           I *rows, V *vals, cudaStream_t st) {
        if (!sa.lean_walk) return false;
        using Kernel = void (*)(GA, TierCommon, I *, V *);
        Kernel k = nullptr;
        switch (T) {
            case 512: k = mode ? k_mid<I, V, 512, 1> : k_mid<I, V, 512, 0>; break;
            case 1024: k = mode ? k_mid<I, V, 1024, 1> : k_mid<I, V, 1024, 0>; break;
            case 2048: k = mode ? k_mid<I, V, 2048, 1> : k_mid<I, V, 2048, 0>; break;
            case 4096: k = mode ? k_mid<I, V, 4096, 1> : k_mid<I, V, 4096, 0>; break;
            case 8192: k = mode ? k_mid<I, V, 8192, 1> : k_mid<I, V, 8192, 0>; break;
            default: k = mode ? k_mid<I, V, 16384, 1> : k_mid<I, V, 16384, 0>; break;
        }
        const int smem = mid_smem<V>(T, thr, mode);
        const int per_sm = std::max(1, std::min(2048 / thr, (227 * 1024) / (smem + 1536)));
        const int want = count < 0 ? cx.nsm * per_sm : count;
        k<<<std::max(1, std::min(want, cx.nsm * per_sm)), thr, smem, st>>>(sa, c, rows, vals);
        return true;
    }

    // count < 0: population unknown on the host (device-driven persistent grid)
    template <class Src>
    static void launch_sym_tier(const Ctx &cx, const typename Src::Args &sa, TierCommon c, int t,
                                int count, cudaStream_t st) {
        c.tier = t;
        const int T = 2 * tier_cap(t);
        if (t <= kWarpTiers) {
            // one warp per column, 8 warps per CTA, warp-private tables
            const int smem = light_smem<V>(T, 0);
            const int per_sm = std::max(1, std::min(8, (228 * 1024) / (smem + 1024)));
            const int want = count < 0 ? cx.nsm * per_sm : (count + 7) / 8;
            const int blocks = std::max(1, std::min(want, cx.nsm * per_sm));
            if constexpr (!Src::kParts) {
                if (sa.lean_walk) {
                    switch (T) {
                        case 64: k_light<I, V, 64, 0><<<blocks, 256, smem, st>>>(sa, c, nullptr, nullptr); break;
                        case 256: k_light<I, V, 256, 0><<<blocks, 256, smem, st>>>(sa, c, nullptr, nullptr); break;
                        case 512: k_light<I, V, 512, 0><<<blocks, 256, smem, st>>>(sa, c, nullptr, nullptr); break;
                        default: k_light<I, V, 1024, 0><<<blocks, 256, smem, st>>>(sa, c, nullptr, nullptr); break;
                    }
                    return;
                }
            }
            switch (T) {
                case 64: k_sym_warp<Src, 64><<<blocks, 256, smem, st>>>(sa, c); break;
                case 256: k_sym_warp<Src, 256><<<blocks, 256, smem, st>>>(sa, c); break;
                case 512: k_sym_warp<Src, 512><<<blocks, 256, smem, st>>>(sa, c); break;
                default: k_sym_warp<Src, 1024><<<blocks, 256, smem, st>>>(sa, c); break;
            }
            return;
        }
        const int thr = block_tier_threads(T, cx.tun);
        c.next_col = cx.cursor + 32 + t;   // zeroed with the cursors at the start of the pass
        if constexpr (!Src::kParts) {
            if (launch_mid(cx, sa, c, T, thr, 0, count, nullptr, nullptr, st)) return;
        }
        const int smem = T * 4;
        const int per_sm = std::max(1, std::min(2048 / thr, (228 * 1024) / (smem + 34 * 1024)));
        const int want = count < 0 ? cx.nsm * per_sm : count;
        const int blocks = std::max(1, std::min(want, cx.nsm * per_sm));
        switch (T) {
            case 512: k_sym_block<Src, 512><<<blocks, thr, smem, st>>>(sa, c); break;
            case 1024: k_sym_block<Src, 1024><<<blocks, thr, smem, st>>>(sa, c); break;
            case 2048: k_sym_block<Src, 2048><<<blocks, thr, smem, st>>>(sa, c); break;
            case 4096: k_sym_block<Src, 4096><<<blocks, thr, smem, st>>>(sa, c); break;
            case 8192: k_sym_block<Src, 8192><<<blocks, thr, smem, st>>>(sa, c); break;
            default: k_sym_block<Src, 16384><<<blocks, thr, smem, st>>>(sa, c); break;
        }
    }

    template <class Src>
    static void launch_num_tier(const Ctx &cx, const typename Src::Args &sa, TierCommon c, int t,
                                int count, I *rows, V *vals, cudaStream_t st) {
        c.tier = t;
        const int T = 2 * tier_cap(t);
        if (t <= kWarpTiers) {
            const int smem = light_smem<V>(T, 1);
            const int per_sm = std::max(1, std::min(8, (228 * 1024) / (smem + 1024)));
            const int want = count < 0 ? cx.nsm * per_sm : (count + 7) / 8;
            const int blocks = std::max(1, std::min(want, cx.nsm * per_sm));
            if constexpr (!Src::kParts) {
                if (sa.lean_walk) {
                    switch (T) {
                        case 64: k_light<I, V, 64, 1><<<blocks, 256, smem, st>>>(sa, c, rows, vals); break;
                        case 256: k_light<I, V, 256, 1><<<blocks, 256, smem, st>>>(sa, c, rows, vals); break;
                        case 512: k_light<I, V, 512, 1><<<blocks, 256, smem, st>>>(sa, c, rows, vals); break;
                        default: k_light<I, V, 1024, 1><<<blocks, 256, smem, st>>>(sa, c, rows, vals); break;
                    }
                    return;
                }
            }
            switch (T) {
                case 64: k_num_warp<Src, 64><<<blocks, 256, smem, st>>>(sa, c, rows, vals); break;
                case 256: k_num_warp<Src, 256><<<blocks, 256, smem, st>>>(sa, c, rows, vals); break;
                case 512: k_num_warp<Src, 512><<<blocks, 256, smem, st>>>(sa, c, rows, vals); break;
                default: k_num_warp<Src, 1024><<<blocks, 256, smem, st>>>(sa, c, rows, vals); break;
            }
            return;
        }
        const int thr = block_tier_threads(T, cx.tun);
        // the tier's column counter: binning cursors 32 + t, zeroed with the
        // cursors at the start of the pass
        c.next_col = cx.cursor + 32 + t;
        if constexpr (!Src::kParts) {
            // The largest tables, unsorted: one CTA of 32 warps per SM, which k_mid's windows of a
            // few dozen B entries do not fill evenly, and no sort to gain on. Numeric tiers, ms, a
            // warp's walk (k_mid) / a CTA's (k_num_block): uniform 500,000 rows, 4,500 a column fp64
            // 7.18 / 6.63, int64 6.58 / 5.93, 150,000 with 7,500 2.57 / 2.56, 2.27 / 2.13; R-MAT of
            // 60,000 rows fp64 1.52 / 1.64 of a step of 12.9. A stage of a k-split keeps k_mid (155 ->
            // 135 us for one of R-MAT 15).
            const bool cta_walk = c.hybrid_sort || (T == 16384 && !c.sort && sa.whole);
            if (!cta_walk && launch_mid(cx, sa, c, T, thr, 1, count, rows, vals, st)) return;
        }
        const int smem = T * (int)(4 + sizeof(V));
        const int per_sm = std::max(1, std::min(2048 / thr, (228 * 1024) / (smem + 34 * 1024)));
        const int want = count < 0 ? cx.nsm * per_sm : count;
        const int blocks = std::max(1, std::min(want, cx.nsm * per_sm));
        switch (T) {
            case 512: k_num_block<Src, 512><<<blocks, thr, smem, st>>>(sa, c, rows, vals); break;
            case 1024: k_num_block<Src, 1024><<<blocks, thr, smem, st>>>(sa, c, rows, vals); break;
            case 2048: k_num_block<Src, 2048><<<blocks, thr, smem, st>>>(sa, c, rows, vals); break;
            case 4096: k_num_block<Src, 4096><<<blocks, thr, smem, st>>>(sa, c, rows, vals); break;
            case 8192: k_num_block<Src, 8192><<<blocks, thr, smem, st>>>(sa, c, rows, vals); break;
            default: k_num_block<Src, 16384><<<blocks, thr, smem, st>>>(sa, c, rows, vals); break;
        }
    }

    static int dense_smem(const Ctx &cx) {
        const int R = 1 << cx.tun.log2R;
        return R * (int)sizeof(V) + R;
    }

    // k_num_heavy32: the accumulator and a presence bitmap
    static int heavy32_smem(const Ctx &cx) {
        const int R = 1 << cx.tun.log2R;
        return R * (int)sizeof(V) + R / 8;
    }

    // largest hash-range item (output rows) whose table (2x slots) fits the
    // memory of a dense item
    static int range_cap(const Ctx &cx) {
        const int R = 1 << cx.tun.log2R;
        const int fit = (int)((int64_t)R * (sizeof(V) + 1) / (sizeof(V) + 4) / 2);
        int cap = 64;
        while (cap * 2 <= fit && cap * 2 <= kRangeCap) cap *= 2;
        return cap;
    }

    // Whether the products of heavy columns run in k_num_heavy32: every entry
    // index < nnz(A) < 2^31 - 8192, and the largest hash table of an item lies inside
    // the accumulator.
    static bool heavy32(const Ctx &cx, const GA &ga) {
        return ga.lean_dense && 2 * range_cap(cx) * (int)(sizeof(V) + 4) <= (1 << cx.tun.log2R) * (int)sizeof(V);
    }

    static int heavy_smem(const Ctx &cx) {
        const int hs = 2 * range_cap(cx) * (int)(sizeof(V) + 4);
        return std::max(dense_smem(cx), hs);
    }

    // Cut the heavy columns of the symbolic list into work items (dense
    // panels and hash ranges) from their per-panel output counts, dense items
    // before hash items, each by first panel. The total and the part of it that
    // columns above cap_full make are left on the device (ioff[0], ioff[1]) and copied
    // to item_total(cx) and full_items(cx), read by the caller after its next wait: with one panel a column has at most one item, so there is room for
    // all before the total is known. Otherwise it is read here, between the
    // count and the items. Few columns and panels take one launch (a product
    // of 3,000 rows spent 55 us on eight launches and two waits).
    // max_panels: panels one hash item may span (any number for the products;
    // kRangeMaxPanels when the items are later sorted, or merged part by part)
    static int64_t item_total(const Ctx &cx) {
        int64_t t;
        std::memcpy(&t, cx.h_small + 256, sizeof(t));
        return t;
    }
    static int64_t full_items(const Ctx &cx) {
        int64_t t;
        std::memcpy(&t, cx.h_small + 258, sizeof(t));
        return t;
    }
    static spgemm_status build_items(const Ctx &cx, int nheavy, const int32_t *sym_list,
                                     const int32_t *sym_off, const int64_t *sel,
                                     const int32_t *pcnt, DevBuf &items, DevBuf &icnt,
                                     DevBuf &ioff, DevBuf &order, cudaStream_t st,
                                     int max_panels = kRangeMaxPanels) {
        std::memset(cx.h_small + 256, 0, 2 * sizeof(int64_t));
        if (!nheavy) return SPGEMM_OK;
        SPG_CK(icnt.ensure(sizeof(int64_t) * (size_t)(std::max(nheavy, cx.P) + 1)));
        SPG_CK(ioff.ensure(sizeof(int64_t) * (nheavy + 1)));
        const int R = 1 << cx.tun.log2R;
        // a panel with at least R/8 output rows is a dense item; the rest are
        // grouped into hash items of at most range_cap rows, so a lone panel
        // below the dense threshold must fit one (dense_min - 1 <= range_cap)
        const int rcap = range_cap(cx);
        const int dmin = std::max(1, std::min(R / 8, rcap));
        int64_t *total_d = ioff.as<int64_t>();
        int32_t *bins = reinterpret_cast<int32_t *>(icnt.p);
        const bool one = (int64_t)nheavy * cx.P <= kItemsOne && 2 * cx.P <= kItemBins;
        const unsigned nb = (unsigned)((nheavy + 255) / 256);
        auto read_total = [&]() {
            return cudaMemcpyAsync(cx.h_small + 256, total_d, 2 * sizeof(int64_t), cudaMemcpyDeviceToHost, st);
        };
        auto run_one = [&](int64_t room) {
            k_heavy_items_one<<<1, 1024, 0, st>>>(sym_list, sym_off, sel, cx.tun.hash_cap_max, cx.cap_full, pcnt, cx.P,
                                                  dmin, rcap, max_panels, room, items.as<HeavyItem>(), order.as<int32_t>(),
                                                  total_d);
            cx.launched();
        };
        auto run_bins = [&](int mode) {
            k_heavy_items<<<nb, 256, 0, st>>>(sym_list, sym_off, sel, cx.tun.hash_cap_max, cx.cap_full, pcnt, cx.P, dmin,
                                              rcap, max_panels, mode, bins, items.as<HeavyItem>(), order.as<int32_t>());
            cx.launched();
        };
        auto size_items = [&](int64_t cnt) -> cudaError_t {
            const cudaError_t e = items.ensure(sizeof(HeavyItem) * (size_t)(cnt + 1));
            return e != cudaSuccess ? e : order.ensure(sizeof(int32_t) * (size_t)(cnt + 1));
        };
        if (cx.P == 1) SPG_CK(size_items(nheavy));
        if (one) {
            run_one(cx.P == 1 ? nheavy : 0);
        } else {
            SPG_CK(cudaMemsetAsync(bins, 0, sizeof(int32_t) * (2 * (size_t)cx.P + 1), st));
            run_bins(0);
            k_small_excl_scan<<<1, 1024, 0, st>>>(bins, 2 * cx.P, total_d);
            cx.launched();
        }
        SPG_CK(read_total());
        if (cx.P > 1) {
            SPG_CK(cudaStreamSynchronize(st));
            SPG_CK(size_items(item_total(cx)));
        }
        if (!one) run_bins(1);
        else if (cx.P > 1) run_one(item_total(cx));
        SPG_CK(cudaGetLastError());
        return SPGEMM_OK;
    }

    // ---- symbolic pass -------------------------------------------------------
    // Bins columns [c_lo, c_hi) of the source, counts distinct rows into
    // cnt_out, fills list/off; heavy columns get per-panel counts in pcnt.
    // heavy_ord_w (optional) receives the heavy ordinals (full pass only).
    // Products: f receives the multiplications per column, total_out their
    // sum, and nnz_b is the number of B entries. recap (optional) may lower or
    // raise the hash cap once the total and the columns above the line (their number and
    // the sums of k_col_tier) are known; the columns are then binned again. zeroed: cx.hist and f are zero already; rows_c: rows of C (products).
    template <class Src>
    static spgemm_status sym_pass(Ctx &cx, const typename Src::Args &sa, int64_t c_lo, int64_t c_hi,
                           const int64_t *bound, int64_t *f, uint8_t *tier, int64_t *cnt_out,
                           int32_t *list, int32_t *off, int32_t *heavy_ord_w,
                           const int32_t *heavy_ord_r, DevBuf *pcnt_grow, int32_t *pcnt_ptr,
                           int *hist_out, cudaStream_t st, bool allow_heavy = true, int64_t nnz_b = 0,
                           int64_t *total_out = nullptr, const std::function<int(int64_t, const Above &)> &recap = nullptr,
                           bool zeroed = false, int64_t rows_c = 0) {
        const int64_t nc = c_hi - c_lo;
        int hist[16];
        int64_t total = 0;
        for (bool again = false;; again = true) {
          const bool small = !Src::kParts && !bound && nc > 0 && nc <= kBinSmall;
          // k_bin_small writes the words that a second binning needs
          if (!(zeroed && !again) && !(small && again))
              SPG_CK(cudaMemsetAsync(cx.hist, 0, sizeof(int32_t) * kBinInts, st));
          if (nc > 0) {
            const int tb = cx.tbegin(kPhFlopsBin, st);
            if (!Src::kParts && !again) {   // all columns of one product
                if (!zeroed) SPG_CK(cudaMemsetAsync(f, 0, sizeof(int64_t) * (size_t)nc, st));
                const int64_t per = 256 * kFlopsEntries;
                if constexpr (!Src::kParts) {
                    if (nnz_b > 0) {
                        k_col_flops<I, V><<<(unsigned)((nnz_b + per - 1) / per), 256, 0, st>>>(
                            sa, nc, reinterpret_cast<unsigned long long *>(f),
                            reinterpret_cast<unsigned long long *>(cx.hist + kFlopTotal));
                        cx.launched();
                    }
                }
            }
            bool binned = false;
            if constexpr (!Src::kParts) {
                if (small) {
                    k_bin_small<<<1, 1024, 0, st>>>(f, rows_c, cx.cap_full, nullptr, nullptr, c_lo, (int)nc,
                                                    cx.tun.hash_cap_max, tier, cnt_out, list, off, heavy_ord_w, cx.hist,
                                                    cx.hist + kOverFull, cx.cursor);
                    binned = true;
                }
            }
            if (!binned) {
                k_col_tier<Src><<<(unsigned)((nc + 255) / 256), 256, 0, st>>>(
                    sa, c_lo, c_hi, cx.tun.hash_cap_max, cx.cap_full, bound, f, tier, cnt_out, cx.hist, cx.hist + kOverFull);
                k_bin_scatter<<<(unsigned)((nc + 255) / 256), 256, 0, st>>>(tier, c_lo, c_hi, cx.hist,
                                                                           cx.cursor, list, off,
                                                                           heavy_ord_w);
            }
            cx.tend(tb, st);
            cx.launched(binned ? 1 : 2);
            SPG_CK(cudaGetLastError());
          }
          SPG_CK(cudaMemcpyAsync(cx.h_small, cx.hist, sizeof(int32_t) * (kAbove + 6), cudaMemcpyDeviceToHost, st));
          SPG_CK(cudaStreamSynchronize(st));
          cx.over_full = cx.h_small[kOverFull];
          std::memcpy(hist, cx.h_small, sizeof(hist));
          if (!again) std::memcpy(&total, cx.h_small + kFlopTotal, sizeof(int64_t));
          Above above;
          for (int t = kHeavyTier0; t < kTiers; ++t) above.n += hist[t];
          std::memcpy(&above.sum, cx.h_small + kAbove, 3 * sizeof(int64_t));
          const int cap = recap && !again ? recap(total, above) : cx.tun.hash_cap_max;
          if (cap == cx.tun.hash_cap_max) break;
          cx.tun.hash_cap_max = cap;
        }
        if (total_out) *total_out = total;
        if (nc <= 0) std::memset(hist, 0, sizeof(hist));
        if (hist_out) std::memcpy(hist_out, hist, sizeof(hist));
        int nheavy = 0;
        for (int t = kHeavyTier0; t < kTiers; ++t) nheavy += hist[t];
        if (nheavy && !allow_heavy) {
            set_error("a column's entries summed over its sources (capped at the row count) exceed " +
                      std::to_string(cx.tun.hash_cap_max) +
                      ", the largest shared-memory hash table this call may use");
            return SPGEMM_ERR_INVALID;
        }
        TierCommon c = common_of(cx);
        c.list = list; c.list_off = off; c.cnt = cnt_out;
        const int th = cx.tbegin(kPhSymHash, st);
        for (int t = 1; t <= 8; ++t)
            if (hist[t]) { launch_sym_tier<Src>(cx, sa, c, t, hist[t], st); cx.launched(); }
        cx.tend(th, st);
        if (nheavy) {
            if (pcnt_grow) {
                SPG_CK(pcnt_grow->ensure(sizeof(int32_t) * (size_t)nheavy * cx.P));
                pcnt_ptr = pcnt_grow->as<int32_t>();
            }
            c.pcnt = pcnt_ptr;
            c.heavy_ord = heavy_ord_r;
            const int64_t items = (int64_t)nheavy * cx.Q;
            const int smem = (int)(((cx.Rs + 31) / 32) * 4);
            const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(items, cx.nsm));
            const int tb = cx.tbegin(kPhSymHeavy, st);
            c.next_col = cx.cursor + 63;   // zeroed with the cursors above
            bool lean = false;
            if constexpr (std::is_same<Src, SrcGemm<I, V>>::value) {
                if (sa.lean_sym) {
                    // CTAs of 512 threads, three or more per SM, where that many
                    // bitmaps fit; one of 1024 threads per SM for wider ones
                    const int per_sm = std::min(4, (227 * 1024) / (smem + (int)sizeof(SymShared<512>) + 1024));
                    if (per_sm >= 3)
                        k_sym_heavy32<I, V, 512, 3><<<(int)std::min<int64_t>(items, (int64_t)cx.nsm * per_sm), 512, smem, st>>>(sa, c);
                    else
                        k_sym_heavy32<I, V, 1024, 1><<<blocks, 1024, smem, st>>>(sa, c);
                    lean = true;
                }
            }
            if (!lean) k_sym_bitmap<Src><<<blocks, 1024, smem, st>>>(sa, c);
            cx.tend(tb, st);
            cx.launched();
        }
        SPG_CK(cudaGetLastError());
        return SPGEMM_OK;
    }

    // ---- numeric pass --------------------------------------------------------
    // tc: host tier populations (nullptr: device-driven grids). heavy: whether
    // dense items exist. sym_list/sym_off: the symbolic heavy list.
    template <class Src, class DSrc, class RSrc = DSrc>
    static spgemm_status num_pass(const Ctx &cx, const typename Src::Args &sa,
                           const typename DSrc::Args &da, int64_t c_lo, int64_t c_hi,
                           const int64_t *cnt, const int64_t *dense_sel, const NumOut<I, V> &o,
                           const int *tc, bool heavy, const int32_t *sym_list,
                           const int32_t *sym_off, const int32_t *heavy_ord,
                           const int32_t *pcnt_in, uint8_t *tier, int32_t *list, int32_t *off,
                           cudaStream_t st, const HeavyItem *items = nullptr, int64_t n_items = 0,
                           const int32_t *item_order = nullptr) {
        const int64_t nc = c_hi - c_lo;
        bool any_hash = tc == nullptr;
        if (tc) for (int t = 1; t <= 8; ++t) any_hash |= tc[t] > 0;
        TierCommon c = common_of(cx);
        c.colptr = o.colptr;
        c.out_base = o.out_base;
        if (any_hash && nc > 0) {
            const int th = cx.tbegin(cx.ph_hash, st);
            if (nc <= kBinSmall) {
                k_bin_small<<<1, 1024, 0, st>>>(nullptr, 0, 0, cnt, dense_sel, c_lo, (int)nc, cx.tun.hash_cap_max, tier,
                                                nullptr, list, off, nullptr, cx.hist, nullptr, cx.cursor);
            } else {
                SPG_CK(cudaMemsetAsync(cx.hist, 0, sizeof(int32_t) * kBinInts, st));
                k_numeric_tier<<<(unsigned)((nc + 255) / 256), 256, 0, st>>>(
                    cnt, dense_sel, c_lo, c_hi, cx.tun.hash_cap_max, tier, cx.hist);
                k_bin_scatter<<<(unsigned)((nc + 255) / 256), 256, 0, st>>>(
                    tier, c_lo, c_hi, cx.hist, cx.cursor, list, off, nullptr);
            }
            SPG_CK(cudaGetLastError());
            c.list = list; c.list_off = off;
            for (int t = 1; t <= 8; ++t) {
                if (tier_cap(t) > cx.tun.hash_cap_max) break;
                const int cntt = tc ? tc[t] : -1;
                if (cntt != 0) { launch_num_tier<Src>(cx, sa, c, t, cntt, o.rows, o.vals, st); cx.launched(); }
            }
            cx.launched(nc <= kBinSmall ? 1 : 2);
            cx.tend(th, st);
        }
        if (heavy) {
            c.list = sym_list; c.list_off = sym_off;
            c.dense_sel = dense_sel;
            c.heavy_ord = heavy_ord;
            c.pcnt_in = pcnt_in;
            c.c_lo = c_lo; c.c_hi = c_hi;
            c.item_counts_from_pcnt = cx.stage_items ? 1 : 0;
            c.range_cap = range_cap(cx);
            if constexpr (!std::is_same<RSrc, DSrc>::value) {
              if (items) {
                // 512-thread CTAs; 3 per SM when the item memory allows it
                // (registers are then capped at 40 per thread), else 2
                using HS = typename HashSrcOf<RSrc>::type;
                const int smem = heavy_smem(cx);
                const int stat = (int)sizeof(BlockShared<V, 512>) + 256;
                const int per_sm = (3 * (smem + stat) <= 227 * 1024) ? 3 : 2;
                const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(n_items, (int64_t)cx.nsm * per_sm));
                if constexpr (std::is_same<RSrc, SrcPanelRange<I, V>>::value) {
                    // products: all heavy items in the kernel with 32-bit offsets
                    if (heavy32(cx, da)) {
                        // three CTAs per SM when their shared memory allows it
                        // (registers are then capped at 40 per thread), else two
                        const int dsm = heavy32_smem(cx);
                        const int dstat = (int)sizeof(DenseShared<V>) + 512;
                        const int dper = std::max(1, std::min(3, (227 * 1024) / (dsm + dstat)));
                        const int dblocks = (int)std::max<int64_t>(1, std::min<int64_t>(n_items, (int64_t)cx.nsm * dper));
                        const int tdd = cx.tbegin(cx.ph_dense, st);
                        // the item counter (the last int of the binning cursors)
                        int *next_item = cx.cursor + 63;
                        SPG_CK(cudaMemsetAsync(next_item, 0, sizeof(int), st));
                        auto kern = cx.sort ? (dper >= 3   ? k_num_heavy32<I, V, 3, true>
                                               : dper == 2 ? k_num_heavy32<I, V, 2, true>
                                                           : k_num_heavy32<I, V, 1, true>)
                                            : (dper >= 3   ? k_num_heavy32<I, V, 3, false>
                                               : dper == 2 ? k_num_heavy32<I, V, 2, false>
                                                           : k_num_heavy32<I, V, 1, false>);
                        kern<<<dblocks, kDenseChunk, dsm, st>>>(da, c, items, item_order, n_items, next_item, o.rows,
                                                                o.vals);
                        cx.tend(tdd, st);
                        cx.launched();
                        SPG_CK(cudaGetLastError());
                        return SPGEMM_OK;
                    }
                }
                const int td = cx.tbegin(cx.ph_dense, st);
                if (per_sm == 3)
                    k_num_heavy<RSrc, HS, 3><<<blocks, 512, smem, st>>>(da, c, items, item_order, n_items,
                                                                        o.rows, o.vals);
                else
                    k_num_heavy<RSrc, HS, 2><<<blocks, 512, smem, st>>>(da, c, items, item_order, n_items,
                                                                        o.rows, o.vals);
                cx.tend(td, st);
                cx.launched();
                SPG_CK(cudaGetLastError());
                return SPGEMM_OK;
              }
            }
            {
                const int smem = dense_smem(cx);
                const int per_sm = std::max(1, std::min(2, (228 * 1024) / (smem + 34 * 1024)));
                const int td = cx.tbegin(cx.ph_dense, st);
                k_num_dense<DSrc><<<cx.nsm * per_sm, 512, smem, st>>>(da, c, o.rows, o.vals);
                cx.tend(td, st);
            }
            cx.launched();
        }
        SPG_CK(cudaGetLastError());
        return SPGEMM_OK;
    }

    // ---- plan ----------------------------------------------------------------
    GA gemm_args(PlanState &ps, int64_t k0, int64_t k1) {
        GA a{};
        a.probs = ps.probs.as<PD>();
        a.nprob = 1;
        a.k0 = k0; a.k1 = k1;
        a.whole = k0 == 0 && k1 == ps.k;
        a.ap_end = ps.ap_end.as<int64_t>();
        a.ap_row = ps.ap_row.as<uint16_t>();
        a.ap_val = ps.ap_val.as<V>();
        a.apc_off = ps.apc_off.as<int32_t>();
        a.apc_row = ps.apc_row.as<uint32_t>();
        a.apc_val = ps.P == 1 ? ps.ap_val.as<V>() : ps.apc_val.as<V>();   // one panel: the same order
        a.lean_dense = narrow(ps) ? 1 : 0;
        a.lean_walk = narrow_walk(ps) ? 1 : 0;
        // a chunk's stream is at most kSymChunk columns of A, each of at most
        // min(m, nnz(A)) entries
        a.lean_sym = a.lean_dense && std::min<int64_t>(ps.A.nrows, ps.A.nnz) * kSymChunk < (int64_t(1) << 31);
        return a;
    }

    // Whether the kernels with 32-bit entry offsets and stream positions may run: a
    // walk looks up to 8192 positions past the stream it is in, and those of light
    // columns as far past the column of B (at most k entries).
    static constexpr int64_t kLeanMost = (int64_t(1) << 31) - 8192;
    static bool narrow(const PlanState &ps) { return ps.A.nnz < kLeanMost; }
    static bool narrow_walk(const PlanState &ps) { return narrow(ps) && ps.k < kLeanMost; }

    // Columns above this many rows are heavy (k_sym_heavy32, k_num_heavy32),
    // unless the caller gave hash_max_cap. The largest table that fits a CTA
    // (8192 rows) is not always the best line: a dense item accumulates without
    // probing, leaves its rows in order, three run per SM against one
    // 1024-thread CTA with the 8192-row table, and one launch takes the place of a launch
    // per tier; but it scans all its rows twice, and the panel copies and item lists are
    // launches of their own (some 45 us). Measured steps, unsorted / sorted, ms, cap 8192
    // -> the lower line:
    //   m in one panel, m / 16, columns of many sizes: fp32 R-MAT of 1,000 rows 0.247 -> 0.208 /
    //     0.262 -> 0.210, of 16,000 1.63 -> 1.22 / 1.81 -> 1.26, protein stand-in of 8,000 rows
    //     0.297 -> 0.224 / 0.317 -> 0.240 (860 products a column above the line); fp64 R-MAT of
    //     8,000 rows 1.18 -> 0.88 / 1.26 -> 0.90; int64 0.84 -> 0.89 / 0.96 -> 0.91;
    //   columns of one size (uniform graphs), one well-filled tier: fp32 5,000 rows with 620
    //     products a column 0.173 -> 0.274 / 0.188 -> 0.307, with 1,400 0.228 -> 0.304 /
    //     0.254 -> 0.300, with 3,500 0.334 -> 0.342 / 0.392 -> 0.337, 10,000 with 2,900
    //     0.587 -> 0.656 / 0.698 -> 0.663, 2,000 with 5,000 0.183 -> 0.200 / 0.192 -> 0.200; but
    //     16,000 with 4,600 1.54 -> 1.13 / 1.83 -> 1.16, fp64 4,000 with 5,900 0.405 -> 0.362 /
    //     0.464 -> 0.366, int64 0.368 -> 0.395 / 0.427 -> 0.398 (lower_pays);
    //   more panels, 4096: fp32 protein stand-in 20,011 / 100,000 columns 1.66 -> 1.49 /
    //     1.96 -> 1.71 and 10.0 -> 9.7 / 12.1 -> 11.8, R-MAT of 60,000 rows 7.24 -> 7.17 /
    //     8.02 -> 7.75; from about 500,000 rows on, the symbolic bitmaps leave one CTA per
    //     SM. With 8-byte values up to two panels (uniform 16,000 with 11,000 products
    //     3.10 -> 2.22 / 3.76 -> 2.24): the panels are half as wide, and a column of a few
    //     thousand rows is cut into as many items (uniform 40,000 with 7,500 rows a column
    //     0.98 -> 1.23 / 1.18 -> 1.23, 500,000 12.6 -> 16.5 / 15.2 -> 19.7, int64 40,000
    //     0.90 -> 1.50 / 1.11 -> 1.51); fp64 columns of many sizes up to eight (R-MAT of 17,000 rows
    //     2.29 -> 1.96 / 2.46 -> 2.06, 40,000 5.78 -> 5.58 / 6.10 -> 5.85, 120,000 22.7 -> 22.6 /
    //     24.6 -> 24.7), int64 ones not (30,000 2.77 -> 2.90 / 3.05 -> 3.09).
    // A k-split keeps 8192 (its stages read every heavy column again: 4-stage R-MAT 15
    // 8.07 -> 8.24 ms), and so does a product that the budget may cut into batches.
    static int heavy_rule(const PlanState &ps) {
        if (!ps.cap_rule || ps.s > 1 || ps.opts.prune || !narrow(ps)) return ps.cap_full;
        if (ps.P == 1) {
            int cap = 256;
            while (cap < ps.cap_full && (int64_t)cap * 16 < ps.m) cap *= 2;
            return cap;
        }
        const int64_t most = int64_t(1) << (sizeof(V) == 4 ? 19 : kIntValue ? 14 : 16);
        return ps.m <= most ? std::min(ps.cap_full, 4096) : ps.cap_full;
    }

    // Whether the columns above the lower line gain by it: their multiplications
    // spread (a variance of log2 of 1/8: a uniform graph's is below 0.08, R-MAT's 0.4 to 2.9,
    // the protein stand-in's 0.17 to 2.3), or they are many on average and in total. Each counts
    // up to kRuleMost and by its logarithm, so that a few hubs do not speak for the rest.
    static constexpr bool kIntValue = std::is_integral<typename Storage<V>::type>::value;
    static bool lower_pays(const PlanState &ps, const Above &a) {
        const double n = (double)a.n, mean = a.n ? (double)a.lg / n : 0.0;
        const bool spread = (double)a.sq - n * mean * mean >= n * (64.0 * 64.0 / 8.0);
        if (sizeof(V) == 8 && ps.m > (int64_t(1) << 14)) return spread;
        return spread || (a.sum >= 4096 * a.n && a.sum >= (int64_t(1) << 24));
    }

    // Whether C fits one batch whatever its columns' overlap is: with as many
    // entries as multiplications, and the heavy columns' workspace at its largest
    // (in place of what an earlier step left of it, so that every symbolic step on
    // a plan decides the same).
    static bool one_batch(const PlanState &ps, int64_t flops) {
        const int64_t si = ps.idx64 ? 8 : 4, sv = sizeof(V), r = si + sv;
        const int64_t inputs = (int64_t)(ps.A.nnz + ps.B.nnz) * r + (ps.A.ncols + ps.B.ncols + 2) * si;
        const int64_t heavy = ps.A.nnz * (2 + 4 + 2 * sv) + ps.k * ((int64_t)ps.P + 1) * 16 +
                              ps.n * ((int64_t)ps.P * 4 + 64) + (1 << 20);
        const int64_t items = ps.P == 1 ? 0 : std::min(ps.n * (int64_t)ps.P, flops) * 28;
        const int ring = ps.opts.ring_depth > 0 ? ps.opts.ring_depth : 2;
        const int64_t other = (int64_t)ps.workspace_bytes() - (int64_t)ps.heavy_bytes();
        return inputs + other + heavy + items + ring * (flops * r + 8 * ps.n) <= (int64_t)ps.budget;
    }

    // The heavy columns' workspace if the line were at cap_full.
    static size_t full_line_bytes(const PlanState &ps) {
        if (ps.over_full == 0) return 0;
        const size_t nh = (size_t)ps.over_full, np = (size_t)ps.P, it = np == 1 ? nh : (size_t)ps.full_items;
        return ps.panel_bytes() + sizeof(int32_t) * nh * np + sizeof(int64_t) * (std::max(nh, np) + 1) +
               sizeof(int64_t) * (nh + 1) + (sizeof(HeavyItem) + sizeof(int32_t)) * (it + 1);
    }

    static bool incremental(const PlanState &ps) {
        return ps.s > 1 && ps.opts.merge_mode == SPGEMM_MERGE_INCREMENTAL;
    }

    spgemm_status setup(PlanState &ps, cudaStream_t st) override {
        attrs();
        PD pd{};
        pd.ap = (const I *)ps.A.colptr; pd.ai = (const I *)ps.A.rowidx; pd.av = (const V *)ps.A.vals;
        pd.bp = (const I *)ps.B.colptr; pd.bi = (const I *)ps.B.rowidx; pd.bv = (const V *)ps.B.vals;
        pd.m = ps.m; pd.gcol0 = 0; pd.ncols = ps.n; pd.ka = ps.k;
        const int64_t n = ps.n;
        const size_t c = (size_t)(n + 1), i64 = sizeof(int64_t), i32 = sizeof(int32_t);
        const size_t stages = ps.s > 1 ? (size_t)ps.s * c : 0;
        SPG_CK(carve<SPGEMM_MEM_DEVICE>(
            ps.arena,
            // err, hist and f are zeroed together; colptr and col_ws are read back
            // together (as h_colptr and h_tier_blk below)
            {{&ps.probs, sizeof(PD)}, {&ps.err, sizeof(int) * 4}, {&ps.hist, i32 * kBinInts}, {&ps.f, i64 * c},
             {&ps.cnt, i64 * c}, {&ps.colptr, i64 * c}, {&ps.col_ws, std::max(i64 * c, i32 * tier_words(ps))},
             {&ps.tier, c + 15}, {&ps.list_sym, i32 * c}, {&ps.list_num, i32 * c}, {&ps.heavy_ord, i32 * c},
             {&ps.off_sym, i32 * 64}, {&ps.off_num, i32 * 64}, {&ps.scan_part, i64 * (size_t)scan_partials_len(n + 1)},
             {&ps.stage_cnt, i64 * stages}, {&ps.stage_colptr, i64 * stages}}));
        SPG_CK(carve<SPGEMM_MEM_PINNED_HOST>(
            ps.h_arena, {{&ps.h_colptr, i64 * c}, {&ps.h_tier_blk, i32 * tier_words(ps)}, {&ps.h_small, 4096},
                         {&ps.h_stage_colptr, i64 * stages}}));
        SPG_CK(cudaMemcpyAsync(ps.probs.p, &pd, sizeof(PD), cudaMemcpyHostToDevice, st));
        SPG_CK(cudaMemsetAsync(ps.err.p, 0, sizeof(int) * 4, st));
        return SPGEMM_OK;
    }

    spgemm_status symbolic(PlanState &ps, cudaStream_t st) override {
        const int64_t n = ps.n;
        ps.have_symbolic = false;
        ps.panels_built = false;
        ps.tun.hash_cap_max = heavy_rule(ps);
        Ctx cx = make_ctx(ps);
        // the error word, the bins and the flops lie next to each other
        SPG_CK(cudaMemsetAsync(ps.err.p, 0, (size_t)((char *)ps.f.p - (char *)ps.err.p) + sizeof(int64_t) * (size_t)(n + 1), st));
        // the rule's cap stays where the columns above it gain by it and the flops
        // bound C to a single batch
        const auto recap = [&](int64_t flops, const Above &above) {
            const bool keep = lower_pays(ps, above) && one_batch(ps, flops);
            return cx.tun.hash_cap_max == ps.cap_full || keep ? cx.tun.hash_cap_max : ps.cap_full;
        };
        // full product: flops, counts, heavy list
        SPG_ST(sym_pass<SrcGemm<I, V>>(cx, gemm_args(ps, 0, ps.k), 0, n, nullptr, ps.f.as<int64_t>(),
                                       ps.tier.as<uint8_t>(), ps.cnt.as<int64_t>(),
                                       ps.list_sym.as<int32_t>(), ps.off_sym.as<int32_t>(),
                                       ps.heavy_ord.as<int32_t>(), ps.heavy_ord.as<int32_t>(),
                                       &ps.pcnt, nullptr, ps.sym_hist, st, true, ps.B.nnz, &ps.flops, recap, true, ps.m));
        ps.tun.hash_cap_max = cx.tun.hash_cap_max;
        ps.over_full = cx.over_full;
        ps.nheavy = 0;
        for (int t = kHeavyTier0; t < kTiers; ++t) ps.nheavy += ps.sym_hist[t];
        const int tsc = cx.tbegin(kPhScan, st);
        SPG_CK(exclusive_scan_i64(ps.cnt.as<int64_t>(), n, ps.colptr.as<int64_t>(),
                                  ps.scan_part.as<int64_t>(), 1, st));
        cx.tend(tsc, st);
        cx.launched(scan_launches(n));
        // k-split stages: per-stage counts nnz(D_t(:, j)) (LocalSymbolic per stage,
        // Algorithm 3), panel counts for the heavy columns
        if (ps.s > 1) {
            if (ps.nheavy)
                SPG_CK(ps.stage_pcnt.ensure(sizeof(int32_t) * (size_t)ps.s * ps.nheavy * ps.P));
            for (int t = 0; t < ps.s; ++t) {
                const int64_t k0 = (int64_t)t * ps.k / ps.s, k1 = (int64_t)(t + 1) * ps.k / ps.s;
                int64_t *scnt = ps.stage_cnt.as<int64_t>() + (size_t)t * (n + 1);
                int32_t *spc = ps.nheavy ? ps.stage_pcnt.as<int32_t>() + (size_t)t * ps.nheavy * ps.P
                                         : nullptr;
                SPG_ST(sym_pass<SrcGemm<I, V>>(cx, gemm_args(ps, k0, k1), 0, n, ps.cnt.as<int64_t>(),
                                               ps.col_ws.as<int64_t>(), ps.tier.as<uint8_t>(), scnt,
                                               ps.list_num.as<int32_t>(), ps.off_num.as<int32_t>(),
                                               nullptr, ps.heavy_ord.as<int32_t>(), nullptr, spc,
                                               nullptr, st, true, ps.B.nnz, nullptr, nullptr, false, ps.m));
                SPG_CK(exclusive_scan_i64(scnt, n, ps.stage_colptr.as<int64_t>() + (size_t)t * (n + 1),
                                          ps.scan_part.as<int64_t>(), 1, st));
                cx.launched(scan_launches(n));
            }
            SPG_CK(cudaMemcpyAsync(ps.h_stage_colptr.p, ps.stage_colptr.p,
                                   sizeof(int64_t) * (size_t)ps.s * (n + 1), cudaMemcpyDeviceToHost, st));
            // incremental merge: counts of the running sums M_u = D_0 + ... + D_u,
            // i.e. the product over k in [0, k1_u), for u = 1..s-2 (M_0 is D_0,
            // M_{s-1} is C), with panel counts for the heavy columns
            if (incremental(ps) && ps.s > 2) {
                const int nu = ps.s - 2;
                SPG_CK(ps.pref_cnt.ensure(sizeof(int64_t) * (size_t)nu * (n + 1)));
                SPG_CK(ps.pref_colptr.ensure(sizeof(int64_t) * (size_t)nu * (n + 1)));
                SPG_CK(ps.h_pref_colptr.ensure(sizeof(int64_t) * (size_t)nu * (n + 1)));
                if (ps.nheavy)
                    SPG_CK(ps.pref_pcnt.ensure(sizeof(int32_t) * (size_t)nu * ps.nheavy * ps.P));
                for (int u = 1; u <= nu; ++u) {
                    const int64_t k1 = (int64_t)(u + 1) * ps.k / ps.s;
                    int64_t *pc = ps.pref_cnt.as<int64_t>() + (size_t)(u - 1) * (n + 1);
                    int32_t *pp = ps.nheavy ? ps.pref_pcnt.as<int32_t>() + (size_t)(u - 1) * ps.nheavy * ps.P
                                            : nullptr;
                    SPG_ST(sym_pass<SrcGemm<I, V>>(cx, gemm_args(ps, 0, k1), 0, n, ps.cnt.as<int64_t>(),
                                                   ps.col_ws.as<int64_t>(), ps.tier.as<uint8_t>(), pc,
                                                   ps.list_num.as<int32_t>(), ps.off_num.as<int32_t>(),
                                                   nullptr, ps.heavy_ord.as<int32_t>(), nullptr, pp,
                                                   nullptr, st, true, ps.B.nnz, nullptr, nullptr, false, ps.m));
                    SPG_CK(exclusive_scan_i64(pc, n, ps.pref_colptr.as<int64_t>() + (size_t)(u - 1) * (n + 1),
                                              ps.scan_part.as<int64_t>(), 1, st));
                    cx.launched(scan_launches(n));
                }
                SPG_CK(cudaMemcpyAsync(ps.h_pref_colptr.p, ps.pref_colptr.p,
                                       sizeof(int64_t) * (size_t)nu * (n + 1), cudaMemcpyDeviceToHost, st));
            }
        }
        SPG_ST(count_tiers(ps, cx, st));
        if (ps.nheavy) SPG_ST(build_panels(ps, st));
        // products alone: a hash item may span any number of panels (one run
        // of the column-grouped copy of A); the items that k_sort_items orders
        // and the k-split's part-by-part merges keep the narrower form
        const int max_panels = (ps.s > 1 || !ps.A.nnz || (ps.opts.sort_output && !heavy32(cx, gemm_args(ps, 0, ps.k))) ||
                                !narrow(ps))
                                   ? kRangeMaxPanels : std::max(kRangeMaxPanels, ps.P);
        SPG_ST(build_items(cx, ps.nheavy, ps.list_sym.as<int32_t>(), ps.off_sym.as<int32_t>(),
                           ps.cnt.as<int64_t>(), ps.pcnt.as<int32_t>(), ps.items, ps.item_cnt,
                           ps.item_off, ps.item_order, st, max_panels));
        SPG_CK(cudaStreamSynchronize(st));
        ps.n_items = item_total(cx);
        ps.full_items = full_items(cx);
        const int errw = ps.h_tier_blk.as<int32_t>()[tier_words(ps) - 1];
        if (errw) {
            set_error("symbolic: device error flags " + std::to_string(errw));
            return SPGEMM_ERR_OVERFLOW;
        }
        ps.nnz_c = ps.h_colptr.as<int64_t>()[n];
        SPG_ST(plan_batches(ps));
        SPG_ST(order_items_by_batch(ps, st));
        if (ps.s > 1) SPG_ST(setup_stage_buffers(ps, st));
        ps.have_symbolic = true;
        return SPGEMM_OK;
    }

    // Order the heavy items batch-major, so that a batch's numeric launch
    // walks its own items only (not every item of the product with a
    // column-range test); inside a batch dense items come first, then hash
    // items, each panel-major. batch_item_off records each batch's run. The
    // item-count buffer is the scratch: without room for the panel histogram
    // the order inside a (batch, kind) is arbitrary, and without room for
    // that the panel-major order of all items stays.
    spgemm_status order_items_by_batch(PlanState &ps, cudaStream_t st) {
        ps.batch_item_off.clear();
        const int64_t nb = (int64_t)ps.batches.size();
        if (!ps.nheavy || ps.n_items <= 0 || nb < 1) return SPGEMM_OK;
        if (nb == 1) {   // built in that order
            ps.batch_item_off = {0, ps.n_items};
            return SPGEMM_OK;
        }
        const int64_t capw = (int64_t)(ps.item_cnt.bytes / sizeof(int64_t));
        const int64_t caps = (int64_t)(ps.scan_part.bytes / sizeof(int64_t));
        auto fits = [&](int64_t pe) {
            const int64_t nbins = nb * 2 * pe;
            return nbins + 1 + nb + 1 <= capw && scan_partials_len(nbins + 1) <= caps;
        };
        const int pe = fits(ps.P) ? ps.P : 1;
        if (!fits(pe)) return SPGEMM_OK;
        const int64_t nbins = nb * 2 * pe;
        unsigned long long *cnt = ps.item_cnt.as<unsigned long long>();
        int64_t *bounds = reinterpret_cast<int64_t *>(cnt + nbins + 1);
        std::vector<int64_t> hb((size_t)nb + 1);
        for (int64_t t = 0; t < nb; ++t) hb[(size_t)t] = ps.batches[(size_t)t].c0;
        hb[(size_t)nb] = ps.batches[(size_t)nb - 1].c1;
        SPG_CK(cudaMemcpyAsync(bounds, hb.data(), sizeof(int64_t) * (size_t)(nb + 1), cudaMemcpyHostToDevice, st));
        SPG_CK(cudaMemsetAsync(cnt, 0, sizeof(int64_t) * (size_t)(nbins + 1), st));
        const unsigned ob = (unsigned)std::max<int64_t>(1, std::min<int64_t>((ps.n_items + 255) / 256, 4096));
        const HeavyItem *items = ps.items.as<HeavyItem>();
        k_items_by_batch<<<ob, 256, 0, st>>>(items, ps.n_items, bounds, nb, pe, 0, cnt, nullptr);
        SPG_CK(exclusive_scan_i64(reinterpret_cast<int64_t *>(cnt), nbins, reinterpret_cast<int64_t *>(cnt),
                                  ps.scan_part.as<int64_t>(), 0, st));
        k_items_by_batch<<<ob, 256, 0, st>>>(items, ps.n_items, bounds, nb, pe, 1, cnt,
                                             ps.item_order.as<int32_t>());
        k_batch_item_starts<<<(unsigned)((nb + 1 + 255) / 256), 256, 0, st>>>(cnt, nb, pe, ps.n_items, bounds);
        ps.timer.launches += 3 + scan_launches(nbins, true);
        SPG_CK(cudaGetLastError());
        std::vector<int64_t> off((size_t)nb + 1);
        SPG_CK(cudaMemcpyAsync(off.data(), bounds, sizeof(int64_t) * (size_t)(nb + 1), cudaMemcpyDeviceToHost, st));
        SPG_CK(cudaStreamSynchronize(st));
        ps.batch_item_off.swap(off);
        return SPGEMM_OK;
    }

    // The heavy items of batch t: its run of item_order when the items are
    // ordered batch-major, else all of them (the kernels skip other columns).
    struct BatchItems {
        int64_t n;
        const int32_t *order;
    };
    static BatchItems batch_items(const PlanState &ps, int64_t t) {
        if (ps.batch_item_off.size() == ps.batches.size() + 1) {
            const int64_t a = ps.batch_item_off[(size_t)t];
            return {ps.batch_item_off[(size_t)t + 1] - a, ps.item_order.as<int32_t>() + a};
        }
        return {ps.n_items, ps.item_order.as<int32_t>()};
    }

    spgemm_status build_panels(PlanState &ps, cudaStream_t st) {
        const int64_t ka = ps.k;
        const int64_t N = (int64_t)ps.P * ka;
        const int64_t nnzA = ps.A.nnz;
        SPG_CK(ps.ap_end.ensure(sizeof(int64_t) * (N + 1)));
        SPG_CK(ps.ap_row.ensure(sizeof(uint16_t) * (nnzA + 8)));
        SPG_CK(ps.ap_val.ensure(sizeof(V) * (nnzA + 8)));
        SPG_CK(ps.merge_tmp.ensure(sizeof(int64_t) * scan_partials_len(N + 1)));
        const int tp = ps.timer.begin(kPhPanels, st);
        SPG_CK(ps.apc_off.ensure(sizeof(int32_t) * (size_t)(ka * ((int64_t)ps.P + 1))));
        SPG_CK(ps.apc_row.ensure(sizeof(uint32_t) * (nnzA + 8)));
        const I *ap = (const I *)ps.A.colptr, *ai = (const I *)ps.A.rowidx;
        int32_t *apo = ps.apc_off.as<int32_t>();
        if (ps.P == 1) {
            const int64_t w = std::max(ka, nnzA);
            k_panel_single<I, V><<<(unsigned)std::max<int64_t>(1, std::min<int64_t>((w + 255) / 256, ps.nsm * 8)), 256, 0, st>>>(
                ap, ai, (const V *)ps.A.vals, ka, ps.ap_end.as<int64_t>(), apo, ps.ap_row.as<uint16_t>(),
                ps.apc_row.as<uint32_t>(), ps.ap_val.as<V>());
            ps.timer.end(tp, st);
            ps.timer.launches += 1;
            SPG_CK(cudaGetLastError());
            ps.panels_built = true;
            return SPGEMM_OK;
        }
        SPG_CK(ps.apc_val.ensure(sizeof(V) * (nnzA + 8)));
        SPG_CK(cudaMemsetAsync(apo, 0, sizeof(int32_t) * (size_t)(ka * ((int64_t)ps.P + 1)), st));
        const unsigned eb = (unsigned)((nnzA + 8 * kPanelWindow - 1) / (8 * kPanelWindow));   // 8 warps per CTA
        if (nnzA > 0)
            k_panel_count<I><<<eb, 256, 0, st>>>(ap, ai, ka, ps.tun.log2R, ps.P, apo);
        const unsigned kb = (unsigned)std::max<int64_t>(1, std::min<int64_t>((ka + 255) / 256, 1 << 20));
        k_panel_starts<<<kb, 256, 0, st>>>(ka, ps.P, apo, ps.ap_end.as<int64_t>());
        SPG_CK(exclusive_scan_i64(ps.ap_end.as<int64_t>(), N, ps.ap_end.as<int64_t>(),
                                  ps.merge_tmp.as<int64_t>(), 0, st));
        if (nnzA > 0)
            k_panel_scatter<I, V><<<eb, 256, 0, st>>>(ap, ai, (const V *)ps.A.vals, ka, ps.tun.log2R, ps.P,
                                                      ps.ap_end.as<unsigned long long>(), apo,
                                                      ps.ap_row.as<uint16_t>(), ps.ap_val.as<V>(),
                                                      ps.apc_row.as<uint32_t>(), ps.apc_val.as<V>());
        ps.timer.end(tp, st);
        ps.timer.launches += (nnzA > 0 ? 3 : 1) + scan_launches(N, true);
        SPG_CK(cudaGetLastError());
        ps.panels_built = true;
        return SPGEMM_OK;
    }

    // The launches of a batch's hash tiers need the tier populations of its
    // columns on the host. k_tier_blocks counts them per block of
    // kTierBlock columns; a batch adds up its whole blocks and looks at
    // single columns only at its two ends. (Counting column by column on the
    // host took 0.25 ms per 50,000 columns, a third of a 2-path count of that
    // size, with the device idle.) Tables: [0] C, then (s > 1) the stages and
    // the running sums M_1..M_{s-2} of the incremental merge.
    static int tier_tables(const PlanState &ps) {
        return ps.s == 1 ? 1 : 1 + ps.s + (incremental(ps) ? ps.s - 2 : 0);
    }
    static int64_t tier_block_count(int64_t n) { return (n + kTierBlock - 1) / kTierBlock; }

    static size_t tier_words(const PlanState &ps) {   // the tables, then the error word
        return (size_t)tier_tables(ps) * (size_t)tier_block_count(ps.n) * 16 + 1;
    }

    // Enqueues the counts and the copy of C's offsets and the counts to the host
    // (the error word last).
    static spgemm_status count_tiers(PlanState &ps, const Ctx &cx, cudaStream_t st) {
        const int64_t n = ps.n, nblk = tier_block_count(n);
        const int nt = tier_tables(ps);
        const size_t words = tier_words(ps);
        int32_t *blk = ps.col_ws.as<int32_t>();   // the stages' flops are no longer needed
        for (int i = 0; i < nt; ++i) {
            const int64_t *cp = i == 0 ? ps.colptr.as<int64_t>()
                                : i <= ps.s ? ps.stage_colptr.as<int64_t>() + (size_t)(i - 1) * (n + 1)
                                            : ps.pref_colptr.as<int64_t>() + (size_t)(i - 1 - ps.s) * (n + 1);
            k_tier_blocks<<<(unsigned)std::max<int64_t>(1, nblk), kTierBlock, 0, st>>>(
                cp, i == 0 ? nullptr : ps.colptr.as<int64_t>(), n, cx.tun.hash_cap_max, blk + (size_t)i * nblk * 16,
                ps.err.as<int>(), blk + words - 1);
        }
        cx.launched(nt);
        SPG_CK(cudaGetLastError());
        // the offsets and the counts behind them, in one copy
        const size_t gap = (size_t)((char *)blk - ps.colptr.as<char>());
        SPG_CK(cudaMemcpyAsync(ps.h_colptr.p, ps.colptr.p, gap + sizeof(int32_t) * words, cudaMemcpyDeviceToHost, st));
        return SPGEMM_OK;
    }

    // Tier populations of columns [c0, c1) from table i of the block counts;
    // cp / sel: the host offsets that the table was counted from.
    static void tier_counts(const PlanState &ps, int i, const int64_t *cp, const int64_t *sel, int64_t c0,
                            int64_t c1, int capmax, std::array<int, 16> &tc, int64_t *heavy) {
        tc.fill(0);
        const int32_t *blk = ps.h_tier_blk.as<int32_t>() + (size_t)i * tier_block_count(ps.n) * 16;
        auto single = [&](int64_t a, int64_t z) {
            for (int64_t j = a; j < z; ++j)
                tc[num_tier(cp[j + 1] - cp[j], sel ? sel[j + 1] - sel[j] : 0, capmax)]++;
        };
        const int64_t b0 = std::min(c1, (c0 + kTierBlock - 1) / kTierBlock * kTierBlock);
        // the last block of the matrix is whole even when it is short
        const int64_t b1 = c1 == ps.n ? c1 : std::max(b0, c1 / kTierBlock * kTierBlock);
        single(c0, b0);
        for (int64_t b = (b0 + kTierBlock - 1) / kTierBlock; b * kTierBlock < b1; ++b)
            for (int t = 0; t < 16; ++t) tc[t] += blk[(size_t)b * 16 + t];
        single(b1, c1);
        if (heavy) *heavy = tc[kHeavyTier0];
        for (int t = kHeavyTier0; t < 16; ++t) tc[t] = 0;
        tc[0] = 0;
    }

    // Greedy contiguous column ranges under the per-batch cap, from the exact
    // per-column counts (Eq. (2)'s smallest b for contiguous ranges).
    spgemm_status plan_batches(PlanState &ps) {
        const int64_t n = ps.n;
        const int64_t *hc = ps.h_colptr.as<int64_t>();
        const int64_t *hs = ps.s > 1 ? ps.h_stage_colptr.as<int64_t>() : nullptr;
        const int64_t r = (ps.idx64 ? 8 : 4) + (ps.vtype == SPGEMM_F32 ? 4 : 8);
        ps.bytes_per_nnz = r;
        const int64_t ptr_bytes = 8;
        const int64_t inputs = (int64_t)(ps.A.nnz + ps.B.nnz) * r +
                               (ps.A.ncols + 1 + ps.B.ncols + 1) * (ps.idx64 ? 8 : 4);
        // columns that only heavy_rule made heavy: the product was shown to fit one
        // batch with their workspace, and the cap per batch is the one of the fixed
        // line, whose workspace for heavy columns is counted here
        const int64_t heavy = (int64_t)(ps.tun.hash_cap_max < ps.cap_full ? full_line_bytes(ps) : ps.heavy_bytes());
        // the stage partial buffers are part of each batch's bytes (w_j counts
        // the unmerged entries), so they are not workspace here; this keeps the
        // plan identical across repeated symbolic calls on one plan
        const int64_t ws = (int64_t)ps.workspace_bytes() - (int64_t)ps.drows.bytes -
                           (int64_t)ps.dvals.bytes - (int64_t)ps.parts_tab.bytes -
                           (int64_t)ps.heavy_bytes() + heavy;
        const int64_t avail = (int64_t)ps.budget - inputs - ws;
        const int ring = ps.opts.ring_depth > 0 ? ps.opts.ring_depth : 2;
        if (avail <= 0) {
            set_error("budget " + std::to_string(ps.budget) + " B does not cover the inputs (" +
                      std::to_string(inputs) + " B) and the workspace (" + std::to_string(ws) + " B)");
            return SPGEMM_ERR_BUDGET;
        }
        const int64_t cap = avail / ring;
        ps.batch_cap = cap;
        ps.batches.clear();
        // unmerged entries up to column j: sum over stages of the stage colptrs
        auto unm = [&](int64_t j) {
            if (!hs) return (int64_t)0;
            int64_t u = 0;
            for (int t = 0; t < ps.s; ++t) u += hs[(size_t)t * (n + 1) + j];
            return u;
        };
        // with opts.prune a batch also holds its pruned copy (at most
        // min(nnz_j, topk) entries per column), its colptr and the prune
        // workspace
        const bool prune = ps.opts.prune != 0;
        if (prune) {
            ps.prune_prefix.assign((size_t)n + 1, 0);
            const int64_t k = ps.opts.prune_topk;
            for (int64_t j = 0; j < n; ++j) {
                const int64_t c = hc[j + 1] - hc[j];
                ps.prune_prefix[(size_t)j + 1] = ps.prune_prefix[(size_t)j] + (k > 0 && c > k ? k : c);
            }
        }
        // incremental merge: the stage buffers of columns [c, x) hold the
        // largest stage partial D_t (t >= 1) and nm running sums, each sized
        // by the largest M_u (u <= s-2; M_0 = D_0)
        const bool inc = incremental(ps);
        const int64_t *hp = (inc && ps.s > 2) ? ps.h_pref_colptr.as<int64_t>() : nullptr;
        const int nm = ps.s > 2 ? 2 : 1;
        auto inc_sizes = [&](int64_t c0, int64_t x, int64_t &dsz, int64_t &msz) {
            dsz = 0;
            for (int t = 1; t < ps.s; ++t)
                dsz = std::max(dsz, hs[(size_t)t * (n + 1) + x] - hs[(size_t)t * (n + 1) + c0]);
            msz = hs[x] - hs[c0];
            for (int u = 1; u <= ps.s - 2; ++u)
                msz = std::max(msz, hp[(size_t)(u - 1) * (n + 1) + x] - hp[(size_t)(u - 1) * (n + 1) + c0]);
        };
        auto wprefix = [&](int64_t j) {
            int64_t w = r * (hc[j] + (inc ? 0 : unm(j))) + ptr_bytes * j;
            if (prune) w += r * ps.prune_prefix[(size_t)j] + (ptr_bytes + kPruneWsPerCol) * j;
            return w;
        };
        // bytes of a batch over columns [c0, x)
        auto wrange = [&](int64_t c0, int64_t x) {
            int64_t w = wprefix(x) - wprefix(c0);
            if (inc) {
                int64_t d, m;
                inc_sizes(c0, x, d, m);
                w += r * (d + nm * m);
            }
            return w;
        };
        int64_t c = 0;
        if (n == 0) {
            Batch b;
            b.tc.resize(ps.s > 1 ? ps.s + 1 : 1);
            for (auto &x : b.tc) x.fill(0);
            ps.batches.push_back(b);
        }
        while (c < n) {
            int64_t lo = c, hi = n;
            while (lo < hi) {
                const int64_t mid = lo + (hi - lo + 1) / 2;
                if (wrange(c, mid) <= cap) lo = mid; else hi = mid - 1;
            }
            if (lo == c) {
                set_error("column " + std::to_string(c) + " needs " + std::to_string(wrange(c, c + 1)) +
                          " B, more than one batch may hold (" + std::to_string(cap) + " B)");
                return SPGEMM_ERR_BUDGET;
            }
            Batch b;
            b.c0 = c; b.c1 = lo; b.nnz = hc[lo] - hc[c];
            b.unmerged = hs ? unm(lo) - unm(c) : b.nnz;
            if (inc) inc_sizes(c, lo, b.dsz, b.msz);
            b.pnnz = prune ? ps.prune_prefix[(size_t)lo] - ps.prune_prefix[(size_t)c] : b.nnz;
            ps.batches.push_back(b);
            c = lo;
        }
        const int capmax = ps.tun.hash_cap_max;
        int64_t total_unm = 0;
        for (auto &b : ps.batches) {
            if (ps.s == 1) {
                b.tc.resize(1);
                tier_counts(ps, 0, hc, nullptr, b.c0, b.c1, capmax, b.tc[0], &b.heavy);
            } else {
                // [0] the final merge, [1 + t] stage t, [s + u] the merge into
                // the running sum M_u (incremental, u = 1..s-2)
                b.tc.resize(ps.s + 1 + (inc ? ps.s - 2 : 0));
                tier_counts(ps, 0, hc, nullptr, b.c0, b.c1, capmax, b.tc[0], &b.heavy);
                b.doff.resize(ps.s);
                int64_t off = 0;
                for (int t = 0; t < ps.s; ++t) {
                    const int64_t *sc = hs + (size_t)t * (n + 1);
                    tier_counts(ps, 1 + t, sc, hc, b.c0, b.c1, capmax, b.tc[1 + t], nullptr);
                    b.doff[t] = off;
                    off += sc[b.c1] - sc[b.c0];
                }
                if (inc)
                    for (int u = 1; u <= ps.s - 2; ++u)
                        tier_counts(ps, ps.s + u, hp + (size_t)(u - 1) * (n + 1), hc, b.c0, b.c1, capmax,
                                    b.tc[ps.s + u], nullptr);
            }
            total_unm += b.unmerged;
        }
        ps.unmerged = ps.s > 1 ? total_unm : ps.nnz_c;
        ps.stage_buffer_nnz = 0;
        if (ps.s > 1)
            for (auto &b : ps.batches)
                ps.stage_buffer_nnz = std::max(ps.stage_buffer_nnz, inc ? b.dsz + nm * b.msz : b.unmerged);
        return SPGEMM_OK;
    }

    // Partial buffers and per-batch part tables for the k-split merge.
    spgemm_status setup_stage_buffers(PlanState &ps, cudaStream_t st) {
        if (incremental(ps)) return setup_incremental_buffers(ps, st);
        int64_t mx = 0;
        for (auto &b : ps.batches) mx = std::max(mx, b.unmerged);
        SPG_CK(ps.drows.ensure(sizeof(I) * (size_t)(mx + 1)));
        SPG_CK(ps.dvals.ensure(sizeof(V) * (size_t)(mx + 1)));
        const size_t nb = ps.batches.size();
        const size_t bytes = sizeof(PartDev<I, V>) * nb * ps.s;
        SPG_CK(ps.parts_tab.ensure(bytes));
        SPG_CK(ps.h_parts.ensure(bytes));
        auto *tab = ps.h_parts.as<PartDev<I, V>>();
        const int64_t *hs = ps.h_stage_colptr.as<int64_t>();
        for (size_t bi = 0; bi < nb; ++bi) {
            const Batch &b = ps.batches[bi];
            for (int t = 0; t < ps.s; ++t) {
                PartDev<I, V> &p = tab[bi * ps.s + t];
                p.colptr = ps.stage_colptr.as<int64_t>() + (size_t)t * (ps.n + 1);
                p.ptr64 = 1;
                p.sub = hs[(size_t)t * (ps.n + 1) + b.c0] - b.doff[t];
                p.rows = ps.drows.as<I>();
                p.vals = ps.dvals.as<V>();
                p.pcnt = ps.nheavy ? ps.stage_pcnt.as<int32_t>() + (size_t)t * ps.nheavy * ps.P : nullptr;
            }
        }
        SPG_CK(cudaMemcpyAsync(ps.parts_tab.p, ps.h_parts.p, bytes, cudaMemcpyHostToDevice, st));
        SPG_CK(cudaStreamSynchronize(st));
        return SPGEMM_OK;
    }

    // Incremental merge: per batch, the stage buffer holds [D | M_a | M_b]:
    // D (dsz entries) takes stage t >= 1, the running sums alternate between
    // M_a and M_b (msz entries each; M_u lives in region u % 2). The part
    // table has two parts per merge step t = 1..s-1: M_{t-1} and D_t.
    spgemm_status setup_incremental_buffers(PlanState &ps, cudaStream_t st) {
        SPG_CK(ps.drows.ensure(sizeof(I) * (size_t)(ps.stage_buffer_nnz + 1)));
        SPG_CK(ps.dvals.ensure(sizeof(V) * (size_t)(ps.stage_buffer_nnz + 1)));
        const size_t nb = ps.batches.size();
        const int ns = ps.s - 1;
        const size_t bytes = sizeof(PartDev<I, V>) * nb * ns * 2;
        SPG_CK(ps.parts_tab.ensure(bytes));
        SPG_CK(ps.h_parts.ensure(bytes));
        auto *tab = ps.h_parts.as<PartDev<I, V>>();
        for (size_t bi = 0; bi < nb; ++bi) {
            const Batch &b = ps.batches[bi];
            for (int t = 1; t <= ns; ++t) {
                const int u = t - 1;
                PartDev<I, V> &pm = tab[(bi * ns + (size_t)u) * 2];
                PartDev<I, V> &pd = tab[(bi * ns + (size_t)u) * 2 + 1];
                pm.colptr = run_colptr(ps, u);
                pm.ptr64 = 1;
                pm.sub = run_hcolptr(ps, u)[b.c0] - run_offset(b, u);
                pm.rows = ps.drows.as<I>();
                pm.vals = ps.dvals.as<V>();
                pm.pcnt = run_pcnt(ps, u);
                pd.colptr = ps.stage_colptr.as<int64_t>() + (size_t)t * (ps.n + 1);
                pd.ptr64 = 1;
                pd.sub = ps.h_stage_colptr.as<int64_t>()[(size_t)t * (ps.n + 1) + b.c0];
                pd.rows = ps.drows.as<I>();
                pd.vals = ps.dvals.as<V>();
                pd.pcnt = ps.nheavy ? ps.stage_pcnt.as<int32_t>() + (size_t)t * ps.nheavy * ps.P : nullptr;
            }
        }
        SPG_CK(cudaMemcpyAsync(ps.parts_tab.p, ps.h_parts.p, bytes, cudaMemcpyHostToDevice, st));
        SPG_CK(cudaStreamSynchronize(st));
        return SPGEMM_OK;
    }
    // the running sum M_u (u <= s-2): device and host colptr, panel counts,
    // and its offset in a batch's stage buffer
    static const int64_t *run_colptr(const PlanState &ps, int u) {
        return u == 0 ? ps.stage_colptr.as<int64_t>()
                      : ps.pref_colptr.as<int64_t>() + (size_t)(u - 1) * (ps.n + 1);
    }
    static const int64_t *run_hcolptr(const PlanState &ps, int u) {
        return u == 0 ? ps.h_stage_colptr.as<int64_t>()
                      : ps.h_pref_colptr.as<int64_t>() + (size_t)(u - 1) * (ps.n + 1);
    }
    static const int32_t *run_pcnt(const PlanState &ps, int u) {
        if (!ps.nheavy) return nullptr;
        return u == 0 ? ps.stage_pcnt.as<int32_t>()
                      : ps.pref_pcnt.as<int32_t>() + (size_t)(u - 1) * ps.nheavy * ps.P;
    }
    static int64_t run_offset(const Batch &b, int u) { return b.dsz + (int64_t)(u & 1) * b.msz; }

    // ---- numeric -------------------------------------------------------------
    spgemm_status numeric(PlanState &ps, int64_t t, spgemm_csc *C, cudaStream_t st) override {
        const Batch &b = ps.batches[(size_t)t];
        const BatchItems bitems = batch_items(ps, t);
        Ctx cx = make_ctx(ps);
        const int64_t n = ps.n;
        const int64_t *hc = ps.h_colptr.as<int64_t>();
        // the pass that writes C (not the stages of a k-split)
        const bool sort = ps.opts.sort_output && !ps.defer_sort;
        if (ps.s == 1) {
            cx.sort = sort;
            NumOut<I, V> o{ps.colptr.as<int64_t>(), hc[b.c0], (I *)C->rowidx, (V *)C->vals};
            GA ga = gemm_args(ps, 0, ps.k);
            SPG_ST((num_pass<SrcGemm<I, V>, SrcPanel<I, V>, SrcPanelRange<I, V>>(
                cx, ga, ga, b.c0, b.c1, ps.cnt.as<int64_t>(), ps.cnt.as<int64_t>(), o, b.tc[0].data(),
                b.heavy > 0, ps.list_sym.as<int32_t>(), ps.off_sym.as<int32_t>(),
                ps.heavy_ord.as<int32_t>(), ps.pcnt.as<int32_t>(), ps.tier.as<uint8_t>(),
                ps.list_num.as<int32_t>(), ps.off_num.as<int32_t>(), st, ps.items.as<HeavyItem>(),
                bitems.n, bitems.order)));
        } else if (incremental(ps)) {
            SPG_ST(numeric_incremental(ps, cx, t, C, st));
        } else {
            const int64_t *hs = ps.h_stage_colptr.as<int64_t>();
            for (int s = 0; s < ps.s; ++s) {
                const int64_t k0 = (int64_t)s * ps.k / ps.s, k1 = (int64_t)(s + 1) * ps.k / ps.s;
                const int64_t *scp = ps.stage_colptr.as<int64_t>() + (size_t)s * (n + 1);
                const int64_t *scnt = ps.stage_cnt.as<int64_t>() + (size_t)s * (n + 1);
                NumOut<I, V> o{scp, hs[(size_t)s * (n + 1) + b.c0] - b.doff[s], ps.drows.as<I>(),
                               ps.dvals.as<V>()};
                GA ga = gemm_args(ps, k0, k1);
                const int32_t *spc = ps.nheavy ? ps.stage_pcnt.as<int32_t>() + (size_t)s * ps.nheavy * ps.P
                                               : nullptr;
                // heavy columns: the merge's work items with this stage's counts,
                // so each stage column is grouped by the ranges the merge reads
                cx.stage_items = true;
                SPG_ST((num_pass<SrcGemm<I, V>, SrcPanel<I, V>, SrcPanelRange<I, V>>(
                    cx, ga, ga, b.c0, b.c1, scnt, ps.cnt.as<int64_t>(), o, b.tc[1 + s].data(),
                    b.heavy > 0, ps.list_sym.as<int32_t>(), ps.off_sym.as<int32_t>(),
                    ps.heavy_ord.as<int32_t>(), spc, ps.tier.as<uint8_t>(), ps.list_num.as<int32_t>(),
                    ps.off_num.as<int32_t>(), st, ps.items.as<HeavyItem>(),
                    bitems.n, bitems.order)));
                cx.stage_items = false;
            }
            // sort-free hash merge of the stage partials (Sec. IV-D)
            cx.ph_hash = kPhMerge;
            cx.ph_dense = kPhMerge;
            cx.sort = sort;
            PA pa{ps.parts_tab.as<PartDev<I, V>>() + (size_t)t * ps.s, ps.s, ps.m};
            NumOut<I, V> o{ps.colptr.as<int64_t>(), hc[b.c0], (I *)C->rowidx, (V *)C->vals};
            SPG_ST((num_pass<SrcParts<I, V>, SrcPartsPanel<I, V>, SrcPartsRange<I, V>>(
                cx, pa, pa, b.c0, b.c1, ps.cnt.as<int64_t>(), ps.cnt.as<int64_t>(), o, b.tc[0].data(),
                b.heavy > 0, ps.list_sym.as<int32_t>(), ps.off_sym.as<int32_t>(),
                ps.heavy_ord.as<int32_t>(), ps.pcnt.as<int32_t>(), ps.tier.as<uint8_t>(),
                ps.list_num.as<int32_t>(), ps.off_num.as<int32_t>(), st, ps.items.as<HeavyItem>(),
                bitems.n, bitems.order)));
        }
        // the hash tiers and k_num_heavy32 write in row order, and so do dense
        // items: what is left are the hash-range items of the other heavy kernel
        if (sort && b.heavy > 0 && !(ps.s == 1 && heavy32(cx, gemm_args(ps, 0, ps.k))))
            SPG_ST(sort_items(cx, ps.colptr.as<int64_t>(), hc[b.c0], b.c0, b.c1, (I *)C->rowidx, (V *)C->vals,
                              ps.items.as<HeavyItem>(), ps.item_off.as<int64_t>(), ps.n_items, st));
        SPG_CK(rebase_colptr(ps.colptr.as<int64_t>() + b.c0, b.c1 - b.c0, C->colptr,
                             C->ptr_type == SPGEMM_I64, st));
        cx.launched();
        return SPGEMM_OK;
    }

    // Incremental k-split of batch bi: stage 0 goes to the running sum M_0;
    // every later stage t goes to D and is hash-merged with M_{t-1} into M_t
    // (into C for the last stage). Each merge is the same two-part merge as
    // the final one, with the counts and panel counts of M_t.
    spgemm_status numeric_incremental(PlanState &ps, Ctx &cx, int64_t bi, spgemm_csc *C, cudaStream_t st) {
        const Batch &b = ps.batches[(size_t)bi];
        const BatchItems bitems = batch_items(ps, bi);
        const int64_t n = ps.n;
        const int64_t *hc = ps.h_colptr.as<int64_t>();
        const int64_t *hs = ps.h_stage_colptr.as<int64_t>();
        const int ph_hash = cx.ph_hash, ph_dense = cx.ph_dense;
        for (int s = 0; s < ps.s; ++s) {
            const int64_t k0 = (int64_t)s * ps.k / ps.s, k1 = (int64_t)(s + 1) * ps.k / ps.s;
            const int64_t *scp = ps.stage_colptr.as<int64_t>() + (size_t)s * (n + 1);
            const int64_t *scnt = ps.stage_cnt.as<int64_t>() + (size_t)s * (n + 1);
            // stage 0 straight into M_0's region, later stages into D (offset 0)
            const int64_t at = s == 0 ? run_offset(b, 0) : 0;
            NumOut<I, V> o{scp, hs[(size_t)s * (n + 1) + b.c0] - at, ps.drows.as<I>(), ps.dvals.as<V>()};
            GA ga = gemm_args(ps, k0, k1);
            const int32_t *spc = ps.nheavy ? ps.stage_pcnt.as<int32_t>() + (size_t)s * ps.nheavy * ps.P
                                           : nullptr;
            cx.ph_hash = ph_hash;
            cx.ph_dense = ph_dense;
            cx.stage_items = true;
            SPG_ST((num_pass<SrcGemm<I, V>, SrcPanel<I, V>, SrcPanelRange<I, V>>(
                cx, ga, ga, b.c0, b.c1, scnt, ps.cnt.as<int64_t>(), o, b.tc[1 + s].data(), b.heavy > 0,
                ps.list_sym.as<int32_t>(), ps.off_sym.as<int32_t>(), ps.heavy_ord.as<int32_t>(), spc,
                ps.tier.as<uint8_t>(), ps.list_num.as<int32_t>(), ps.off_num.as<int32_t>(), st,
                ps.items.as<HeavyItem>(), bitems.n, bitems.order)));
            if (s == 0) continue;
            // M_s = M_{s-1} + D_s (sort-free hash merge, Sec. IV-D)
            cx.ph_hash = kPhMerge;
            cx.ph_dense = kPhMerge;
            PA pa{ps.parts_tab.as<PartDev<I, V>>() + ((size_t)bi * (ps.s - 1) + (size_t)(s - 1)) * 2, 2, ps.m};
            if (s < ps.s - 1) {
                const int64_t *mcp = run_colptr(ps, s);
                const int64_t *mcnt = ps.pref_cnt.as<int64_t>() + (size_t)(s - 1) * (n + 1);
                NumOut<I, V> om{mcp, run_hcolptr(ps, s)[b.c0] - run_offset(b, s), ps.drows.as<I>(),
                                ps.dvals.as<V>()};
                cx.stage_items = true;
                SPG_ST((num_pass<SrcParts<I, V>, SrcPartsPanel<I, V>, SrcPartsRange<I, V>>(
                    cx, pa, pa, b.c0, b.c1, mcnt, ps.cnt.as<int64_t>(), om, b.tc[ps.s + s].data(),
                    b.heavy > 0, ps.list_sym.as<int32_t>(), ps.off_sym.as<int32_t>(),
                    ps.heavy_ord.as<int32_t>(), run_pcnt(ps, s), ps.tier.as<uint8_t>(),
                    ps.list_num.as<int32_t>(), ps.off_num.as<int32_t>(), st, ps.items.as<HeavyItem>(),
                    bitems.n, bitems.order)));
            } else {
                NumOut<I, V> oc{ps.colptr.as<int64_t>(), hc[b.c0], (I *)C->rowidx, (V *)C->vals};
                cx.stage_items = false;
                cx.sort = ps.opts.sort_output && !ps.defer_sort;
                SPG_ST((num_pass<SrcParts<I, V>, SrcPartsPanel<I, V>, SrcPartsRange<I, V>>(
                    cx, pa, pa, b.c0, b.c1, ps.cnt.as<int64_t>(), ps.cnt.as<int64_t>(), oc, b.tc[0].data(),
                    b.heavy > 0, ps.list_sym.as<int32_t>(), ps.off_sym.as<int32_t>(),
                    ps.heavy_ord.as<int32_t>(), ps.pcnt.as<int32_t>(), ps.tier.as<uint8_t>(),
                    ps.list_num.as<int32_t>(), ps.off_num.as<int32_t>(), st, ps.items.as<HeavyItem>(),
                    bitems.n, bitems.order)));
            }
        }
        cx.stage_items = false;
        return SPGEMM_OK;
    }

    // ---- sorted output and prune ---------------------------------------------
    // Sort the hash-range items of the heavy columns in [c0, c1) of a batch in
    // place. colptr: the plan's global offsets, base = offset of column c0.
    static spgemm_status sort_items(const Ctx &cx, const int64_t *colptr, int64_t base, int64_t c0,
                                    int64_t c1, I *rows, V *vals, const HeavyItem *items,
                                    const int64_t *nitems_dev, int64_t n_items, cudaStream_t st) {
        if (n_items > 0) {
            // staging for the largest hash item (range_cap rows), a bitmap
            // over item row ranges of up to 16 panels and its 16-bit word
            // prefix (wider ranges fall back to the bitonic sort); two CTAs
            // per SM when that fits
            const int64_t want = (int64_t)kRangeMaxPanels << cx.tun.log2R >> 5;
            auto launch = [&](auto cap_tag) -> void {
                constexpr int CAP = decltype(cap_tag)::value;
                const int stage = (int)(CAP * (4 + sizeof(V)));
                const int fit2 = 110 * 1024;   // bytes per CTA for two CTAs per SM
                const int64_t room = std::max<int64_t>(fit2 - stage, 64 * 1024 - stage);
                const int wcap = (int)std::max<int64_t>(32, std::min<int64_t>(want, room / 6));
                const unsigned ib = (unsigned)std::max<int64_t>(1, std::min<int64_t>(n_items, (int64_t)cx.nsm * 2));
                k_sort_items<I, V, CAP><<<ib, 512, stage + 6 * wcap, st>>>(items, nitems_dev, colptr, base, c0,
                                                                            c1, cx.tun.log2R, wcap, rows, vals);
            };
            if (range_cap(cx) <= 4096) launch(std::integral_constant<int, 4096>{});
            else launch(std::integral_constant<int, 8192>{});
        }
        cx.launched();
        SPG_CK(cudaGetLastError());
        return SPGEMM_OK;
    }

    // The smallest value of type V that is >= thr (so that "v >= it" in V is
    // exactly "v >= thr" in double).
    static V typed_threshold(double thr) {
        using S = typename Storage<V>::type;
        S t;
        if constexpr (std::is_same<S, float>::value) {
            t = (float)thr;
            if (std::isfinite(thr) && (double)t < thr) t = std::nextafterf(t, INFINITY);
        } else if constexpr (std::is_same<S, double>::value) {
            t = thr;
        } else {
            if (thr <= -9.2233720368547758e18) t = INT64_MIN;
            else if (thr > 9.2233720368547748e18) t = INT64_MAX;
            else t = (int64_t)std::ceil(thr);
        }
        if constexpr (std::is_same<V, S>::value) return t;
        else return V::raw(t);
    }

    // bytes per column that the batch plan sets aside for the prune workspace
    // (PruneWs: keep and sel 8 B, mode 1 B, and the scan partials; an upper bound)
    static constexpr int64_t kPruneWsPerCol = 40;

    // Prune step 1: kept count per column, the selections, and out_colptr =
    // exclusive scan of the counts (ncols + 1 entries, total last).
    static spgemm_status prune_plan(const int64_t *colptr, const V *vals, int64_t ncols, V thr, int64_t topk,
                                    PruneWs &ws, int64_t *out_colptr, cudaStream_t st) {
        SPG_CK(ws.ensure(ncols));
        SPG_CK(cudaMemsetAsync(ws.nsel.p, 0, 2 * sizeof(unsigned long long), st));
        if (ncols > 0) {
            const unsigned wb = (unsigned)std::max<int64_t>(1, std::min<int64_t>((ncols + 7) / 8, 1 << 20));
            k_prune_count<V><<<wb, 256, 0, st>>>(colptr, vals, ncols, thr, topk, ws.keep.as<int64_t>(),
                                                 ws.mode.as<int8_t>(), ws.sel.as<int64_t>(),
                                                 ws.nsel.as<unsigned long long>());
        }
        SPG_CK(exclusive_scan_i64(ws.keep.as<int64_t>(), ncols, out_colptr, ws.part.as<int64_t>(), 1, st));
        SPG_CK(cudaGetLastError());
        return SPGEMM_OK;
    }

    // Prune step 2: the kept entries, in input order, at out_colptr.
    template <class IO>
    static spgemm_status prune_fill(const int64_t *colptr, const I *rows, const V *vals, int64_t ncols, V thr,
                                    int64_t topk, int tie_by_row, PruneWs &ws, const int64_t *out_colptr, IO *orows,
                                    V *ovals, int nsm, cudaStream_t st) {
        if (ncols <= 0) return SPGEMM_OK;
        const unsigned wb = (unsigned)std::max<int64_t>(1, std::min<int64_t>((ncols + 7) / 8, 1 << 20));
        k_prune_compact<I, V, IO><<<wb, 256, 0, st>>>(colptr, rows, vals, ncols, thr, ws.mode.as<int8_t>(), out_colptr,
                                                      orows, ovals);
        if (topk > 0) {
            // 100 KB of staged keys: two CTAs of 512 threads per SM
            const int bytes = 100 * 1024, cap = bytes / (KeyBits<V>::v / 8);
            k_prune_select<I, V, IO><<<(unsigned)nsm * 2, kPruneThreads, bytes, st>>>(
                colptr, rows, vals, thr, topk, ws.sel.as<int64_t>(), ws.nsel.as<unsigned long long>(), tie_by_row, cap,
                out_colptr, orows, ovals);
        }
        SPG_CK(cudaGetLastError());
        return SPGEMM_OK;
    }

    // spgemm_prune on a caller's CSC (two-call protocol).
    static spgemm_status prune(const spgemm_csc *in, double thr_d, int64_t topk, spgemm_csc *out,
                               cudaStream_t st) {
        attrs();
        int dev = 0, nsm = 148;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        const int64_t n = in->ncols;
        const V thr = typed_threshold(thr_d);
        DevBuf cp64;
        const int64_t *cp = (const int64_t *)in->colptr;
        if (in->ptr_type == SPGEMM_I32) {
            SPG_CK(cp64.ensure(sizeof(int64_t) * (size_t)(n + 1)));
            k_widen<int32_t><<<(unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 256) / 256, 1 << 20)), 256, 0, st>>>(
                (const int32_t *)in->colptr, n + 1, cp64.as<int64_t>());
            cp = cp64.as<int64_t>();
        }
        PruneWs ws;
        CallScratch scratch(ws.arena, st);
        DevBuf tmp;
        const bool count_only = out->rowidx == nullptr;
        int64_t *ocp = (int64_t *)out->colptr;
        if (!count_only) {   // recount into scratch; out->colptr holds the first call's offsets
            SPG_CK(tmp.ensure(sizeof(int64_t) * (size_t)(n + 1)));
            ocp = tmp.as<int64_t>();
        }
        SPG_ST(prune_plan(cp, (const V *)in->vals, n, thr, topk, ws, ocp, st));
        if (count_only) {
            int64_t total = 0;
            SPG_CK(cudaMemcpyAsync(&total, ocp + n, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
            SPG_CK(cudaStreamSynchronize(st));
            out->nnz = total;
            return SPGEMM_OK;
        }
        const int64_t *fin = (const int64_t *)out->colptr;
        SPG_ST(prune_fill<I>(cp, (const I *)in->rowidx, (const V *)in->vals, n, thr, topk, 0, ws, fin,
                             (I *)out->rowidx, (V *)out->vals, nsm, st));
        SPG_CK(cudaStreamSynchronize(st));   // the scratch buffers go out of scope
        return SPGEMM_OK;
    }

    spgemm_status prune_batch(PlanState &ps, int64_t ncols, const int64_t *colptr, const void *rows,
                              const void *vals, int64_t *ocolptr, void *orows, void *ovals, PruneWs &ws,
                              cudaStream_t st) override {
        const V thr = typed_threshold(ps.opts.prune_threshold);
        // sorted output with a small topk: prune the unsorted batch (ties to
        // the smaller rows, the order sorting would give), then sort only
        // the kept entries
        const int tie_by_row = ps.defer_sort ? 1 : 0;
        const int64_t topk = ps.opts.prune_topk;
        SPG_ST(prune_plan(colptr, (const V *)vals, ncols, thr, topk, ws, ocolptr, st));
        SPG_ST(prune_fill<I>(colptr, (const I *)rows, (const V *)vals, ncols, thr, topk, tie_by_row, ws, ocolptr,
                             (I *)orows, (V *)ovals, ps.nsm, st));
        ps.timer.launches += (ncols <= 0 ? 0 : topk > 0 ? 3 : 2) + scan_launches(ncols);
        if (ps.defer_sort && ncols > 0) {
            // columns of up to 256 kept entries by a warp, 1024 and 8192 by a CTA
            const unsigned wbk = (unsigned)std::max<int64_t>(1, std::min<int64_t>((ncols + 7) / 8, (int64_t)ps.nsm * 8));
            const unsigned bb = (unsigned)std::max<int64_t>(1, std::min<int64_t>(ncols, (int64_t)ps.nsm * 4));
            const int slot = 4 + (int)sizeof(V);
            k_sort_cols<I, V, 512, false><<<wbk, 256, 8 * 512 * slot, st>>>(ocolptr, ncols, 0, (I *)orows, (V *)ovals);
            if (topk > 256)
                k_sort_cols<I, V, 2048, true><<<bb, 512, 2048 * slot, st>>>(ocolptr, ncols, 256, (I *)orows, (V *)ovals);
            if (topk > 1024)
                k_sort_cols<I, V, 16384, true><<<bb, 512, 16384 * slot, st>>>(ocolptr, ncols, 1024, (I *)orows,
                                                                             (V *)ovals);
            ps.timer.launches += 1 + (topk > 256) + (topk > 1024);
            SPG_CK(cudaGetLastError());
        }
        return SPGEMM_OK;
    }

    // ---- backward ------------------------------------------------------------
    spgemm_status backward(PlanState &ps, const spgemm_csc *G, void *dA, void *dB,
                           cudaStream_t st) override {
        if (ps.vtype == SPGEMM_INT64) {
            set_error("backward needs floating-point values");
            return SPGEMM_ERR_INVALID;
        }
        if (IsMinPlus<V>::v || IsOrAnd<V>::v) {
            set_error("backward is defined for the plus-times semiring only");
            return SPGEMM_ERR_INVALID;
        }
        Ctx cx = make_ctx(ps);
        cx.tun.hash_cap_max = ps.cap_full;   // tiers by G's columns, not the product's heavy rule
        const int64_t n = ps.n;
        GradArgs<I, V> ga{};
        ga.gemm = gemm_args(ps, 0, ps.k);
        ga.gcolptr = G->colptr;
        ga.gptr64 = G->ptr_type == SPGEMM_I64;
        ga.grows = (const I *)G->rowidx;
        ga.gvals = (const V *)G->vals;
        ga.dA = (V *)dA;
        ga.dB = (V *)dB;
        const int tbw = cx.tbegin(kPhBackward, st);
        if (ps.A.nnz)
            k_fill_zero<V><<<(unsigned)((ps.A.nnz + 255) / 256), 256, 0, st>>>((V *)dA, ps.A.nnz);
        if (ps.B.nnz)
            k_fill_zero<V><<<(unsigned)((ps.B.nnz + 255) / 256), 256, 0, st>>>((V *)dB, ps.B.nnz);
        cx.launched((ps.A.nnz > 0) + (ps.B.nnz > 0));
        if (n == 0) { cx.tend(tbw, st); return SPGEMM_OK; }
        SPG_CK(cudaMemsetAsync(cx.hist, 0, sizeof(int32_t) * kBinInts, st));
        k_bwd_tier<I, V><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(ga, n, cx.tun.hash_cap_max,
                                                                       ps.tier.as<uint8_t>(), cx.hist);
        k_bin_scatter<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(
            ps.tier.as<uint8_t>(), 0, n, cx.hist, cx.cursor, ps.list_num.as<int32_t>(),
            ps.off_num.as<int32_t>(), nullptr);
        SPG_CK(cudaMemcpyAsync(cx.h_small, cx.hist, sizeof(int32_t) * 16, cudaMemcpyDeviceToHost, st));
        SPG_CK(cudaStreamSynchronize(st));
        int hist[16];
        std::memcpy(hist, cx.h_small, sizeof(hist));
        TierCommon c = common_of(cx);
        c.list = ps.list_num.as<int32_t>();
        c.list_off = ps.off_num.as<int32_t>();
        for (int t = 1; t <= 8; ++t) {
            if (!hist[t]) continue;
            c.tier = t;
            const int T = 2 * tier_cap(t);
            if (t <= kWarpTiers) {
                const bool lean = ga.gemm.lean_walk != 0;
                const int smem = 8 * T * (int)(4 + sizeof(V)) + (lean ? 8 * 32 * (int)(8 + sizeof(V)) : 0);
                const int per_sm = std::max(1, std::min(8, (228 * 1024) / (smem + 1024)));
                const int blocks = std::max(1, std::min((hist[t] + 7) / 8, cx.nsm * per_sm));
                if (lean) {
                    switch (T) {
                        case 64: k_bwd_light<I, V, 64><<<blocks, 256, smem, st>>>(ga, c); break;
                        case 256: k_bwd_light<I, V, 256><<<blocks, 256, smem, st>>>(ga, c); break;
                        case 512: k_bwd_light<I, V, 512><<<blocks, 256, smem, st>>>(ga, c); break;
                        default: k_bwd_light<I, V, 1024><<<blocks, 256, smem, st>>>(ga, c); break;
                    }
                    continue;
                }
                switch (T) {
                    case 64: k_bwd_warp<I, V, 64><<<blocks, 256, smem, st>>>(ga, c); break;
                    case 256: k_bwd_warp<I, V, 256><<<blocks, 256, smem, st>>>(ga, c); break;
                    case 512: k_bwd_warp<I, V, 512><<<blocks, 256, smem, st>>>(ga, c); break;
                    default: k_bwd_warp<I, V, 1024><<<blocks, 256, smem, st>>>(ga, c); break;
                }
                continue;
            }
            const int thr = block_tier_threads(T, cx.tun);
            const int smem = T * (int)(4 + sizeof(V));
            const int per_sm = std::max(1, std::min(2048 / thr, (228 * 1024) / (smem + 34 * 1024)));
            const int blocks = std::max(1, std::min(hist[t], cx.nsm * per_sm));
            switch (T) {
                case 512: k_bwd_block<I, V, 512><<<blocks, thr, smem, st>>>(ga, c); break;
                case 1024: k_bwd_block<I, V, 1024><<<blocks, thr, smem, st>>>(ga, c); break;
                case 2048: k_bwd_block<I, V, 2048><<<blocks, thr, smem, st>>>(ga, c); break;
                case 4096: k_bwd_block<I, V, 4096><<<blocks, thr, smem, st>>>(ga, c); break;
                case 8192: k_bwd_block<I, V, 8192><<<blocks, thr, smem, st>>>(ga, c); break;
                default: k_bwd_block<I, V, 16384><<<blocks, thr, smem, st>>>(ga, c); break;
            }
        }
        int nheavy = 0;
        for (int t = kHeavyTier0; t < kTiers; ++t) nheavy += hist[t];
        if (nheavy) {
            const int smem = dense_smem(cx);
            k_bwd_dense<I, V><<<cx.nsm, 1024, smem, st>>>(ga, c);
            cx.launched();
        }
        for (int t = 1; t <= 8; ++t) if (hist[t]) cx.launched();
        cx.launched(2);
        cx.tend(tbw, st);
        SPG_CK(cudaGetLastError());
        return SPGEMM_OK;
    }

    // ---- standalone merge (spgemm_merge) ---------------------------------------
    static spgemm_status merge(const spgemm_csc *parts, int nparts, spgemm_csc *out, cudaStream_t st) {
        attrs();
        const int64_t n = parts[0].ncols, m = parts[0].nrows;
        int dev = 0, nsm = 0;
        SPG_CK(cudaGetDevice(&dev));
        SPG_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
        PlanState tmp;   // scratch only
        tmp.nsm = nsm;
        tmp.tun.log2R = sizeof(V) == 4 ? 14 : 13;
        const int64_t R = 1ll << tmp.tun.log2R;
        tmp.P = (int)std::max<int64_t>(1, (m + R - 1) / R);
        const int64_t maxbm = (int64_t)(160 * 1024) * 8;
        const int64_t mpad = ((m + R - 1) / R) * R;
        tmp.Rs = mpad <= maxbm ? (mpad > 0 ? mpad : R) : (maxbm / R) * R;
        tmp.Q = (int)std::max<int64_t>(1, (m + tmp.Rs - 1) / tmp.Rs);
        struct Guard { PlanState &p; ~Guard() { p.release_all(); } } guard{tmp};
        CallScratch scratch(tmp.arena, st);
        std::vector<PartDev<I, V>> tab(nparts);
        for (int i = 0; i < nparts; ++i) {
            tab[i].colptr = parts[i].colptr;
            tab[i].ptr64 = parts[i].ptr_type == SPGEMM_I64;
            tab[i].sub = 0;
            tab[i].rows = (const I *)parts[i].rowidx;
            tab[i].vals = (const V *)parts[i].vals;
            tab[i].pcnt = nullptr;
        }
        const size_t c = (size_t)(n + 1), i64 = sizeof(int64_t), i32 = sizeof(int32_t);
        SPG_CK(carve<SPGEMM_MEM_DEVICE>(
            tmp.arena,
            {{&tmp.parts_tab, sizeof(PartDev<I, V>) * (size_t)nparts}, {&tmp.cnt, i64 * c}, {&tmp.colptr, i64 * c},
             {&tmp.tier, c + 15}, {&tmp.list_sym, i32 * c}, {&tmp.list_num, i32 * c}, {&tmp.heavy_ord, i32 * c},
             {&tmp.hist, i32 * kBinInts}, {&tmp.off_sym, i32 * 64}, {&tmp.off_num, i32 * 64},
             {&tmp.err, sizeof(int) * 4}, {&tmp.scan_part, i64 * (size_t)scan_partials_len(n + 1)}}));
        SPG_CK(tmp.h_small.ensure(4096));
        SPG_CK(cudaMemcpyAsync(tmp.parts_tab.p, tab.data(), sizeof(PartDev<I, V>) * nparts,
                               cudaMemcpyHostToDevice, st));
        SPG_CK(cudaMemsetAsync(tmp.err.p, 0, sizeof(int) * 4, st));
        Ctx cx = make_ctx(tmp);
        PA pa{tmp.parts_tab.as<PartDev<I, V>>(), nparts, m};
        int hist[16];
        SPG_ST(sym_pass<SrcParts<I, V>>(cx, pa, 0, n, nullptr, nullptr, tmp.tier.as<uint8_t>(),
                                        tmp.cnt.as<int64_t>(), tmp.list_sym.as<int32_t>(),
                                        tmp.off_sym.as<int32_t>(), tmp.heavy_ord.as<int32_t>(),
                                        tmp.heavy_ord.as<int32_t>(), &tmp.pcnt, nullptr, hist, st));
        SPG_CK(exclusive_scan_i64(tmp.cnt.as<int64_t>(), n, tmp.colptr.as<int64_t>(),
                                  tmp.scan_part.as<int64_t>(), 1, st));
        int64_t nnz = 0;
        SPG_CK(cudaMemcpyAsync(&nnz, tmp.colptr.as<int64_t>() + n, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
        SPG_CK(cudaStreamSynchronize(st));
        if (out->ptr_type == SPGEMM_I32 && nnz > 0x7fffffffLL) {
            set_error("merged nnz does not fit a 32-bit colptr");
            return SPGEMM_ERR_INDEX_OVERFLOW;
        }
        if (!out->rowidx) {
            SPG_CK(rebase_colptr(tmp.colptr.as<int64_t>(), n, out->colptr, out->ptr_type == SPGEMM_I64, st));
            out->nnz = nnz;
            SPG_CK(cudaStreamSynchronize(st));
            return SPGEMM_OK;
        }
        if (out->nnz != nnz) {
            set_error("out->nnz does not match the merged size");
            return SPGEMM_ERR_INVALID;
        }
        int nheavy = 0;
        for (int t = kHeavyTier0; t < kTiers; ++t) nheavy += hist[t];
        SPG_ST(build_items(cx, nheavy, tmp.list_sym.as<int32_t>(), tmp.off_sym.as<int32_t>(),
                           tmp.cnt.as<int64_t>(), tmp.pcnt.as<int32_t>(), tmp.items, tmp.item_cnt,
                           tmp.item_off, tmp.item_order, st));
        SPG_CK(cudaStreamSynchronize(st));
        const int64_t n_items = item_total(cx);
        NumOut<I, V> o{tmp.colptr.as<int64_t>(), 0, (I *)out->rowidx, (V *)out->vals};
        SPG_ST((num_pass<SrcParts<I, V>, SrcPartsPanel<I, V>, SrcPartsRange<I, V>>(
            cx, pa, pa, 0, n, tmp.cnt.as<int64_t>(), tmp.cnt.as<int64_t>(), o, nullptr, nheavy > 0,
            tmp.list_sym.as<int32_t>(), tmp.off_sym.as<int32_t>(), tmp.heavy_ord.as<int32_t>(),
            tmp.pcnt.as<int32_t>(), tmp.tier.as<uint8_t>(), tmp.list_num.as<int32_t>(),
            tmp.off_num.as<int32_t>(), st, tmp.items.as<HeavyItem>(),
            n_items, tmp.item_order.as<int32_t>())));
        int errw = 0;
        SPG_CK(cudaMemcpyAsync(&errw, tmp.err.p, sizeof(int), cudaMemcpyDeviceToHost, st));
        SPG_CK(cudaStreamSynchronize(st));
        if (errw) {
            set_error("merge: device error flags " + std::to_string(errw));
            return SPGEMM_ERR_OVERFLOW;
        }
        return SPGEMM_OK;
    }

    // ---- merge into caller-free scratch (spgemm_merge_noalloc) ----------------
    // Same two-call protocol and kernels as merge(), with every work buffer
    // carved from the given device scratch and host staging in static memory;
    // no allocation of any kind. Columns must fit the shared-memory hash tiers.
    static size_t merge_noalloc_bytes(int64_t n, int nparts) {
        auto al = [](size_t x) { return (x + 255) / 256 * 256; };
        return al(sizeof(int64_t) * (n + 1)) * 2 + al(n + 16) + al(sizeof(int32_t) * (n + 1)) * 3 +
               al(sizeof(int32_t) * kBinInts) + al(sizeof(int32_t) * 64) * 2 + al(sizeof(int) * 4) +
               al(sizeof(int64_t) * scan_partials_len(n + 1)) + al(sizeof(PartDev<I, V>) * nparts);
    }

    static spgemm_status merge_noalloc(const spgemm_csc *parts, int nparts, spgemm_csc *out,
                                       cudaStream_t st, unsigned char *scratch, size_t cap,
                                       int32_t *h_stage, int nsm) {
        const int64_t n = parts[0].ncols, m = parts[0].nrows;
        const size_t need = merge_noalloc_bytes(n, nparts);
        attrs();
        if (need > cap) {
            set_error("merge_noalloc: " + std::to_string(n) + " columns and " + std::to_string(nparts) +
                      " parts need " + std::to_string(need) + " B of scratch; the static scratch holds " +
                      std::to_string(cap) + " B");
            return SPGEMM_ERR_INVALID;
        }
        auto al = [](size_t x) { return (x + 255) / 256 * 256; };
        unsigned char *p = scratch;
        auto take = [&](size_t bytes) { unsigned char *q = p; p += al(bytes); return q; };
        int64_t *cnt = (int64_t *)take(sizeof(int64_t) * (n + 1));
        int64_t *colptr = (int64_t *)take(sizeof(int64_t) * (n + 1));
        uint8_t *tier = (uint8_t *)take(n + 16);
        int32_t *list_sym = (int32_t *)take(sizeof(int32_t) * (n + 1));
        int32_t *list_num = (int32_t *)take(sizeof(int32_t) * (n + 1));
        int32_t *heavy_ord = (int32_t *)take(sizeof(int32_t) * (n + 1));
        int32_t *hist = (int32_t *)take(sizeof(int32_t) * kBinInts);
        int32_t *off_sym = (int32_t *)take(sizeof(int32_t) * 64);
        int32_t *off_num = (int32_t *)take(sizeof(int32_t) * 64);
        int *err = (int *)take(sizeof(int) * 4);
        int64_t *part_sc = (int64_t *)take(sizeof(int64_t) * scan_partials_len(n + 1));
        PartDev<I, V> *tab_d = (PartDev<I, V> *)take(sizeof(PartDev<I, V>) * nparts);
        PartDev<I, V> tab[64];
        for (int i = 0; i < nparts; ++i) {
            tab[i].colptr = parts[i].colptr;
            tab[i].ptr64 = parts[i].ptr_type == SPGEMM_I64;
            tab[i].sub = 0;
            tab[i].rows = (const I *)parts[i].rowidx;
            tab[i].vals = (const V *)parts[i].vals;
            tab[i].pcnt = nullptr;
        }
        // the scratch keeps the previous call's contents: clear what is read
        // before it is written (error word; tier histogram and cursors are
        // cleared inside the passes)
        SPG_CK(cudaMemcpyAsync(tab_d, tab, sizeof(PartDev<I, V>) * nparts, cudaMemcpyHostToDevice, st));
        SPG_CK(cudaMemsetAsync(err, 0, sizeof(int) * 4, st));
        Ctx cx;
        cx.nsm = nsm;
        cx.err = err; cx.hist = hist; cx.cursor = hist + 64; cx.h_small = h_stage;
        cx.tun.log2R = sizeof(V) == 4 ? 14 : 13;
        cx.P = 1; cx.Q = 1; cx.Rs = 32;
        PA pa{tab_d, nparts, m};
        int hist_h[16];
        // columns above the largest hash table would need the dense path's
        // per-panel workspace: sym_pass rejects them before any launch
        SPG_ST(sym_pass<SrcParts<I, V>>(cx, pa, 0, n, nullptr, nullptr, tier, cnt, list_sym, off_sym,
                                        heavy_ord, heavy_ord, nullptr, nullptr, hist_h, st, false));
        SPG_CK(exclusive_scan_i64(cnt, n, colptr, part_sc, 1, st));
        int64_t nnz = 0;
        SPG_CK(cudaMemcpyAsync(&nnz, colptr + n, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
        SPG_CK(cudaStreamSynchronize(st));
        if (out->ptr_type == SPGEMM_I32 && nnz > 0x7fffffffLL) {
            set_error("merged nnz does not fit a 32-bit colptr");
            return SPGEMM_ERR_INDEX_OVERFLOW;
        }
        if (!out->rowidx) {
            SPG_CK(rebase_colptr(colptr, n, out->colptr, out->ptr_type == SPGEMM_I64, st));
            out->nnz = nnz;
            SPG_CK(cudaStreamSynchronize(st));
            return SPGEMM_OK;
        }
        if (out->nnz != nnz) {
            set_error("out->nnz does not match the merged size");
            return SPGEMM_ERR_INVALID;
        }
        NumOut<I, V> o{colptr, 0, (I *)out->rowidx, (V *)out->vals};
        SPG_ST((num_pass<SrcParts<I, V>, SrcPartsPanel<I, V>>(
            cx, pa, pa, 0, n, cnt, cnt, o, nullptr, false, list_sym, off_sym, heavy_ord, nullptr, tier,
            list_num, off_num, st)));
        int errw = 0;
        SPG_CK(cudaMemcpyAsync(&errw, err, sizeof(int), cudaMemcpyDeviceToHost, st));
        SPG_CK(cudaStreamSynchronize(st));
        if (errw) {
            set_error("merge_noalloc: device error flags " + std::to_string(errw));
            return SPGEMM_ERR_OVERFLOW;
        }
        return SPGEMM_OK;
    }

    // ---- many independent products (spgemm_multi) ------------------------------
    static Ctx multi_ctx(MultiState &ms) {
        Ctx c;
        c.nsm = ms.nsm; c.tun = ms.tun; c.err = ms.err.as<int>();
        c.hist = ms.hist.as<int32_t>(); c.cursor = c.hist + 64;
        c.h_small = ms.h_small.as<int32_t>();
        c.P = 1; c.Q = 1; c.Rs = 32;
        return c;
    }

    static GA multi_args(MultiState &ms) {
        GA a{};
        a.probs = ms.probs.as<PD>();
        a.nprob = ms.nprob;
        a.prob_of = ms.prob_of.as<int32_t>();
        a.k0 = 0; a.k1 = INT64_MAX;
        return a;
    }

    static spgemm_status multi_create(MultiState &ms, const spgemm_csc *As, const spgemm_csc *Bs,
                                      cudaStream_t st) {
        attrs();
        std::vector<PD> tab(ms.nprob);
        int64_t g = 0;
        for (int i = 0; i < ms.nprob; ++i) {
            PD &p = tab[i];
            p.ap = (const I *)As[i].colptr; p.ai = (const I *)As[i].rowidx; p.av = (const V *)As[i].vals;
            p.bp = (const I *)Bs[i].colptr; p.bi = (const I *)Bs[i].rowidx; p.bv = (const V *)Bs[i].vals;
            p.m = As[i].nrows; p.gcol0 = g; p.ncols = Bs[i].ncols; p.ka = As[i].ncols;
            g += Bs[i].ncols;
        }
        ms.total_cols = g;
        const int64_t n = g;
        SPG_CK(ms.probs.ensure(sizeof(PD) * ms.nprob));
        SPG_CK(cudaMemcpyAsync(ms.probs.p, tab.data(), sizeof(PD) * ms.nprob, cudaMemcpyHostToDevice, st));
        SPG_CK(ms.f.ensure(sizeof(int64_t) * (n + 1)));
        SPG_CK(ms.cnt.ensure(sizeof(int64_t) * (n + 1)));
        SPG_CK(ms.colptr.ensure(sizeof(int64_t) * (n + 1)));
        SPG_CK(ms.tier.ensure(n + 16));
        SPG_CK(ms.prob_of.ensure(sizeof(int32_t) * (n + 1)));
        SPG_CK(ms.list.ensure(sizeof(int32_t) * (n + 1)));
        SPG_CK(ms.off.ensure(sizeof(int32_t) * 64));
        SPG_CK(ms.hist.ensure(sizeof(int32_t) * kBinInts));
        SPG_CK(ms.err.ensure(sizeof(int) * 4));
        SPG_CK(ms.scan_part.ensure(sizeof(int64_t) * scan_partials_len(n + 1)));
        SPG_CK(ms.h_small.ensure(4096));
        SPG_CK(cudaMemsetAsync(ms.err.p, 0, sizeof(int) * 4, st));
        // flops of every column: arena capacity (nnz <= flops) and tier check
        Ctx cx = multi_ctx(ms);
        SPG_CK(cudaMemsetAsync(cx.hist, 0, sizeof(int32_t) * 64, st));
        if (n > 0)
            k_multi_bin<I, V><<<(unsigned)((n * kBinLanes + 255) / 256), 256, 0, st>>>(
                multi_args(ms), n, cx.tun.hash_cap_max, ms.prob_of.as<int32_t>(), ms.f.as<int64_t>(),
                ms.tier.as<uint8_t>(), ms.cnt.as<int64_t>(), cx.hist);
        SPG_CK(cudaGetLastError());
        SPG_CK(exclusive_scan_i64(ms.f.as<int64_t>(), n, ms.colptr.as<int64_t>(),
                                  ms.scan_part.as<int64_t>(), 1, st));
        SPG_CK(cudaMemcpyAsync(ms.h_small.p, cx.hist, sizeof(int32_t) * 16, cudaMemcpyDeviceToHost, st));
        SPG_CK(cudaMemcpyAsync(ms.h_small.as<char>() + 256, ms.colptr.as<int64_t>() + n, sizeof(int64_t),
                               cudaMemcpyDeviceToHost, st));
        SPG_CK(cudaStreamSynchronize(st));
        int hist[16];
        std::memcpy(hist, ms.h_small.p, sizeof(hist));
        ms.total_flops = *(int64_t *)(ms.h_small.as<char>() + 256);
        ms.capacity = ms.total_flops;
        SPG_CK(ms.rows.ensure(sizeof(I) * (size_t)(ms.capacity + 1)));
        SPG_CK(ms.vals.ensure(sizeof(V) * (size_t)(ms.capacity + 1)));
        // columns above the largest shared-memory table: one global-memory
        // hash table each (2 * min(f_j, m) slots, a power of two)
        ms.heavy_cols = 0;
        for (int t = kHeavyTier0; t < kTiers; ++t) ms.heavy_cols += n > 0 ? hist[t] : 0;
        SPG_CK(ms.gtab_off.ensure(sizeof(int64_t) * (n + 1)));
        if (ms.heavy_cols) {
            SPG_CK(ms.gsize.ensure(sizeof(int64_t) * (n + 1)));
            k_multi_gtab_sizes<SrcGemm<I, V>><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(
                multi_args(ms), ms.f.as<int64_t>(), ms.tier.as<uint8_t>(), n, ms.gsize.as<int64_t>());
            SPG_CK(cudaGetLastError());
            SPG_CK(exclusive_scan_i64(ms.gsize.as<int64_t>(), n, ms.gtab_off.as<int64_t>(),
                                      ms.scan_part.as<int64_t>(), 1, st));
            int64_t gslots = 0;
            SPG_CK(cudaMemcpyAsync(&gslots, ms.gtab_off.as<int64_t>() + n, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
            SPG_CK(cudaStreamSynchronize(st));
            SPG_CK(ms.gkeys.ensure(sizeof(uint32_t) * (size_t)(gslots + 1)));
            SPG_CK(ms.gvals.ensure(sizeof(V) * (size_t)(gslots + 1)));
        }
        SPG_CK(ms.counter.ensure(sizeof(unsigned long long) * 4));
        // shared memory of the persistent passes: the largest CTA table or
        // the warps' private tables, whichever is larger; the symbolic pass needs
        // the keys only, so more of its CTAs are resident
        const size_t nw = (size_t)ms.threads / 32;
        for (int mode = 0; mode < 2; ++mode) {
            const size_t slot = 4 + (mode ? sizeof(V) : 0);
            ms.smem[mode] = std::max((size_t)2 * ms.tun.hash_cap_max, nw * 2 * tier_cap(ms.warp_tiers)) * slot;
            int per_sm = 0;
            SPG_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, multi_kernel(ms.threads, mode), ms.threads,
                                                                 ms.smem[mode]));
            if (per_sm < 1) {
                set_error("the batched tables do not fit shared memory: lower hash_max_cap or warp_max_cap");
                return SPGEMM_ERR_INVALID;
            }
            ms.grid[mode] = ms.nsm * per_sm;
        }
        ms.enqueue = &multi_enqueue;
        return SPGEMM_OK;
    }

    using MultiKernel = void (*)(GA, TierCommon, MultiQueue, I *, V *);
    static MultiKernel multi_kernel(int threads, int mode) {
        if (threads == 512) return mode ? k_multi_pass<SrcGemm<I, V>, 512, 1> : k_multi_pass<SrcGemm<I, V>, 512, 0>;
        if (threads == 256) return mode ? k_multi_pass<SrcGemm<I, V>, 256, 1> : k_multi_pass<SrcGemm<I, V>, 256, 0>;
        return mode ? k_multi_pass<SrcGemm<I, V>, 128, 1> : k_multi_pass<SrcGemm<I, V>, 128, 0>;
    }

    // flops, symbolic, scan and numeric for all problems; no host
    // synchronisation (device-driven tier grids), so it can be captured.
    static spgemm_status multi_enqueue(MultiState &ms, cudaStream_t st) {
        Ctx cx = multi_ctx(ms);
        const int64_t n = ms.total_cols;
        GA ga = multi_args(ms);
        SPG_CK(cudaMemsetAsync(cx.hist, 0, sizeof(int32_t) * kBinInts, st));
        SPG_CK(cudaMemsetAsync(ms.counter.p, 0, sizeof(unsigned long long) * 4, st));
        if (n > 0) {
            // tiers by the flop bound min(f_j, m), the same as at creation
            k_multi_bin<I, V><<<(unsigned)((n * kBinLanes + 255) / 256), 256, 0, st>>>(
                ga, n, cx.tun.hash_cap_max, ms.prob_of.as<int32_t>(), nullptr, ms.tier.as<uint8_t>(),
                ms.cnt.as<int64_t>(), cx.hist);
            k_bin_scatter<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(
                ms.tier.as<uint8_t>(), 0, n, cx.hist, cx.cursor, ms.list.as<int32_t>(),
                ms.off.as<int32_t>(), nullptr);
        }
        TierCommon c = common_of(cx);
        c.cnt = ms.cnt.as<int64_t>();
        MultiQueue mq{ms.list.as<int32_t>(), ms.off.as<int32_t>(), ms.counter.as<unsigned long long>(),
                      ms.gtab_off.as<int64_t>(), ms.gkeys.as<uint32_t>(), ms.gvals.p, ms.warp_tiers};
        // one persistent launch counts every column of every problem ...
        if (n > 0) multi_kernel(ms.threads, 0)<<<ms.grid[0], ms.threads, ms.smem[0], st>>>(ga, c, mq, nullptr, nullptr);
        SPG_CK(cudaGetLastError());
        SPG_CK(exclusive_scan_i64(ms.cnt.as<int64_t>(), n, ms.colptr.as<int64_t>(),
                                  ms.scan_part.as<int64_t>(), 1, st));
        // ... and one forms them, into the output arena at the scanned offsets
        c.colptr = ms.colptr.as<int64_t>();
        c.out_base = 0;
        mq.counter = ms.counter.as<unsigned long long>() + 2;
        if (n > 0)
            multi_kernel(ms.threads, 1)<<<ms.grid[1], ms.threads, ms.smem[1], st>>>(ga, c, mq, ms.rows.as<I>(),
                                                                                    ms.vals.as<V>());
        SPG_CK(cudaGetLastError());
        return SPGEMM_OK;
    }
};

}  // namespace spg
