// Light columns of a product, one warp each, with a warp-private hash table in
// shared memory (C(:, j) = A * B(:, j), Sec. II-C's column formula): the
// symbolic count and the numeric accumulation, with 32-bit entry offsets (the
// caller guarantees nnz(A) and the inner dimension < 2^31 less the look-ahead of a walk).
//
// A column of some hundred products is a chain of dependent loads (column
// list, colptr of B, its rows, colptr of A, A's entries) around little work, so
// the kernels are bound by that latency and by the warps the tables leave
// room for. The chain is spread over the column before: its list entry is read
// two columns ahead, the colptr of B when the previous column starts, B's rows
// after that column's walk and the colptr of A after its output. Measured against
// one chain per column (symbolic / numeric, us): 2-path counts of 200,000 vertices
// with 4 entries a column 103 / 155 -> 75 / 132, uniform 100,000 columns of 11 84 / 174
// -> 67 / 158, 2-path counts 50,021 x 16 97 / 316 -> 81 / 289. What is left is issue:
// some 240 warp instructions per 32 products, the compare-and-swap loops of
// the inserts and of the value adds first (issue slots 40 to 53% busy, a quarter to
// half of the warps resident beside the tables).
#pragma once

namespace spg {

// Dynamic shared memory of k_light: 8 tables and 8 segment lists.
template <class V> constexpr int light_smem(int T, int mode) {
    return 8 * (T + 32) * (4 + (mode == 1 ? (int)sizeof(V) : 0));
}

// CTAs per SM that the registers are fitted to (0: the compiler's choice): what the large
// numeric tables leave room for, so that the walk is not spilled for CTAs that cannot come
// (1024 int64 slots: 80 registers instead of 64 and 36 bytes spilled, numeric tiers of 77,906
// vertices' 2-path counts 634 -> 611 us). Fewer for 512 8-byte slots costs more than the spills
// (50,021 vertices 272 us, 303 with 3).
template <class V> constexpr int light_min_ctas(int T, int mode) {
    return mode == 0 ? 0 : T == 1024 ? 3 : T == 512 && sizeof(V) == 4 ? 5 : 0;
}

// MODE 0: symbolic (c.cnt[g]); MODE 1: numeric, rows in table order or
// ascending (c.sort).
template <class I, class V, int T, int MODE>
__global__ void __launch_bounds__(256, light_min_ctas<V>(T, MODE))
    k_light(GemmArgs<I, V> ga, TierCommon c, I *out_rows, V *out_vals) {
    constexpr int LOG2T = Log2<T>::v;
    constexpr int U = 4;   // windows whose loads are in flight
    // how a lane finds its segment: a shuffle search over the lanes, or one
    // OR-reduce of the segment starts and a table in shared memory (fewer
    // instructions; the large numeric tables gain from the registers instead)
    constexpr bool kSearch = MODE == 1 && T >= 512;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    V *vals = MODE == 1 ? reinterpret_cast<V *>(smem) + warp * T : nullptr;
    uint32_t *keys = reinterpret_cast<uint32_t *>(smem + (MODE == 1 ? sizeof(V) * 8 * T : 0)) + warp * T;
    // per warp: the non-empty segments of a round, in stream order
    unsigned char *segs = smem + (size_t)8 * T * (4 + (MODE == 1 ? sizeof(V) : 0));
    V *s_bv = reinterpret_cast<V *>(segs) + warp * 32;
    int *s_off = reinterpret_cast<int *>(segs + (MODE == 1 ? 8 * 32 * sizeof(V) : 0)) + warp * 32;
    const ProbDev<I, V> *pd = ga.probs;
    const I *bp = pd->bp, *bi = pd->bi, *ap = pd->ap, *ai = pd->ai;
    const V *bv = pd->bv, *av = pd->av;
    const int64_t k0 = ga.k0, k1 = ga.k1;
    const unsigned below = (1u << lane) - 1u, upto = 0xffffffffu >> (31 - lane);
    const int hi = c.list_off[c.tier + 1];
    const int stride = gridDim.x * 8;
    int it = c.list_off[c.tier] + blockIdx.x * 8 + warp;
    if (it >= hi) return;
    // the segment of A that B entry e holds
    auto segment = [&](int64_t k, bool any, int &beg, int &len) {
        beg = 0;
        len = 0;
        if (any && k >= k0 && k < k1) {
            const int64_t a = (int64_t)__ldg(&ap[k]);
            beg = (int)a;
            len = (int)((int64_t)__ldg(&ap[k + 1]) - a);
        }
    };
    int g = c.list[it];
    int gn = it + stride < hi ? c.list[it + stride] : -1;
    int64_t b0 = (int64_t)__ldg(&bp[g]);
    int nb = (int)((int64_t)__ldg(&bp[g + 1]) - b0);
    int64_t k = lane < nb ? (int64_t)__ldg(&bi[b0 + lane]) : 0;
    V bval = V(0);
    if (MODE == 1 && lane < nb) bval = __ldg(&bv[b0 + lane]);
    int beg, len;
    segment(k, lane < nb, beg, len);
    // the table is cleared once; a column's output leaves it clean
    for (int s = lane; s < T; s += 32) {
        keys[s] = kEmpty;
        if (MODE == 1) vals[s] = V(0);
    }
    __syncwarp();
    for (;;) {
        const int64_t b0n = gn >= 0 ? (int64_t)__ldg(&bp[gn]) : 0;
        const int64_t b1n = gn >= 0 ? (int64_t)__ldg(&bp[gn + 1]) : 0;
        const int gnn = it + 2 * (int64_t)stride < hi ? c.list[it + 2 * stride] : -1;
        int64_t o0 = 0, o1 = 0;
        if (MODE == 1) { o0 = c.colptr[g]; o1 = c.colptr[g + 1]; }
        int mine = 0;
        for (int base = 0;;) {
            // the segments of these 32 entries, one per lane, as a stream [0, tot)
            const int incl = warp_incl_scan(len);
            const int excl = incl - len;
            const int tot = __shfl_sync(SPG_FULL, incl, 31);
            const int off = beg - excl;   // stream position + off = entry index
            if (!kSearch) {
                // the non-empty segments in stream order
                const unsigned nzm = __ballot_sync(SPG_FULL, len > 0);
                if (len > 0) {
                    const int rank = __popc(nzm & below);
                    s_off[rank] = off;
                    if (MODE == 1) s_bv[rank] = bval;
                }
                __syncwarp();
            }
            int before = -1;   // segments started before the window, minus one
            for (int w = 0; w < tot; w += 32 * U) {
                uint32_t r[U];
                V x[U];
                bool ok[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int p = w + 32 * u + lane;
                    ok[u] = p < tot;
                    int q;
                    V vs;
                    if (kSearch) {
                        // the last lane whose segment starts at or before p
                        int sl = 0;
#pragma unroll
                        for (int b = 16; b > 0; b >>= 1) {
                            const int e = __shfl_sync(SPG_FULL, excl, sl + b);
                            if (e <= p) sl += b;
                        }
                        q = __shfl_sync(SPG_FULL, off, sl) + p;
                        if (MODE == 1) vs = shfl_bits(bval, sl);
                    } else {
                        // the segments started before the window plus the starts
                        // at or below the lane
                        const unsigned d = (unsigned)(excl - (w + 32 * u));
                        const unsigned M = __reduce_or_sync(SPG_FULL, len > 0 && d < 32u ? 1u << d : 0u);
                        const int sl = before + __popc(M & upto);
                        before += __popc(M);
                        q = ok[u] ? s_off[sl] + p : 0;
                        if (MODE == 1 && ok[u]) vs = s_bv[sl];
                    }
                    if (ok[u]) {
                        r[u] = (uint32_t)__ldg(&ai[q]);
                        if (MODE == 1) x[u] = mul_v(__ldg(&av[q]), vs);
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (!ok[u]) continue;
                    bool nw;
                    const int h = hash_insert_dbl1(keys, LOG2T, r[u], c.err, nw);
                    if (MODE == 0) mine += nw;
                    else if (h >= 0) atomic_add_v(&vals[h], x[u]);
                }
            }
            base += 32;
            if (base >= nb) break;
            if (!kSearch) __syncwarp();   // the segments are read: the next round may replace them
            const bool any = base + lane < nb;
            k = any ? (int64_t)__ldg(&bi[b0 + base + lane]) : 0;
            if (MODE == 1 && any) bval = __ldg(&bv[b0 + base + lane]);
            segment(k, any, beg, len);
        }
        // the next column's rows of B, on their way during this one's output
        b0 = b0n;
        nb = (int)(b1n - b0n);
        k = lane < nb ? (int64_t)__ldg(&bi[b0 + lane]) : 0;
        if (MODE == 1 && lane < nb) bval = __ldg(&bv[b0 + lane]);
        __syncwarp();
        if (MODE == 0) {
            mine = warp_sum(mine);
            if (lane == 0) c.cnt[g] = mine;
            uint4 *k4 = reinterpret_cast<uint4 *>(keys);
            for (int s = lane; s < T / 4; s += 32) k4[s] = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
        } else {
            const int64_t out0 = o0 - c.out_base;
            const int want = (int)(o1 - o0);
            if (c.sort) {
                sorted_emit<false>(keys, vals, T, want, nullptr, c.err, out_rows + out0, out_vals + out0);
            } else {
                int pos = 0;
                for (int s0 = 0; s0 < T; s0 += 32) {
                    const int s = s0 + lane;
                    const uint32_t key = keys[s];
                    const bool occ = key != kEmpty;
                    const unsigned bal = __ballot_sync(SPG_FULL, occ);
                    if (occ) {
                        const int r = pos + __popc(bal & below);
                        if (r < want) {
                            out_rows[out0 + r] = (I)key;
                            out_vals[out0 + r] = vals[s];
                        }
                        keys[s] = kEmpty;
                        vals[s] = V(0);
                    }
                    pos += __popc(bal);
                }
                if (lane == 0 && pos != want) atomicOr(c.err, kErrCount);
            }
        }
        if (gn < 0) return;
        segment(k, lane < nb, beg, len);
        g = gn;
        gn = gnn;
        it += stride;
        __syncwarp();
    }
}

// A warp's part of the products of one column with k in [k0, k1): of the rounds of
// 32 B entries it takes r0, r0 + rs, ..., and of the 32-wide windows of a round's
// product stream w0, w0 + ws, ...; insert(row, product) for each, with the loads of
// four windows in flight. Stream positions are 32-bit: the runs of a column of a
// hash tier have at most as many entries as the column (rows are distinct in a
// column of A), or nnz(A) is below 2^31 less the look-ahead. off / sbv: 32 places
// per warp in shared memory for the non-empty segments of a round, in stream order
// (offset to the entry index, B value). All lanes call it.
template <int MODE, class I, class V, class F>
__device__ __forceinline__ void walk_entries(const ProbDev<I, V> *p, int64_t k0, int64_t k1, int64_t b0, int nb,
                                             int r0, int rs, int w0, int ws, int64_t *off, V *sbv, F &&insert) {
    constexpr int U = 4;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u, upto = 0xffffffffu >> (31 - lane);
    const I *bi = p->bi, *ap = p->ap, *ai = p->ai;
    const V *bv = p->bv, *av = p->av;
    for (int base = 32 * r0; base < nb; base += 32 * rs) {
        int64_t beg = 0;
        int len = 0;
        V bval = V(0);
        if (base + lane < nb) {
            const int64_t k = (int64_t)__ldg(&bi[b0 + base + lane]);
            if (k >= k0 && k < k1) {
                beg = (int64_t)__ldg(&ap[k]);
                len = (int)((int64_t)__ldg(&ap[k + 1]) - beg);
            }
            if (MODE == 1) bval = __ldg(&bv[b0 + base + lane]);
        }
        const int incl = warp_incl_scan(len);
        const int excl = incl - len;
        const int tot = __shfl_sync(SPG_FULL, incl, 31);
        const unsigned nzm = __ballot_sync(SPG_FULL, len > 0);
        if (len > 0) {
            const int rank = __popc(nzm & below);
            off[rank] = beg - excl;
            if (MODE == 1) sbv[rank] = bval;
        }
        __syncwarp();
        for (int w = 32 * w0; w < tot; w += 32 * U * ws) {
            uint32_t r[U];
            V x[U];
            bool ok[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                // the segment of a lane: the last one starting at or before it
                const int wu = w + 32 * u * ws;
                const unsigned d = (unsigned)(excl - wu);
                const unsigned M = __reduce_or_sync(SPG_FULL, len > 0 && d < 32u ? 1u << d : 0u);
                const int before = __popc(__ballot_sync(SPG_FULL, len > 0 && excl < wu));
                const int sl = before + __popc(M & upto) - 1;
                ok[u] = wu + lane < tot;
                if (ok[u]) {
                    const int64_t q = off[sl] + wu + lane;
                    r[u] = (uint32_t)__ldg(&ai[q]);
                    if (MODE == 1) x[u] = mul_v(__ldg(&av[q]), sbv[sl]);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (ok[u]) insert(r[u], MODE == 1 ? x[u] : V(0));
        }
        __syncwarp();   // the segments are read: the next round may replace them
    }
}

// Columns of the CTA tiers (tables of up to 16384 slots), one CTA each, taken
// from a device counter: the symbolic count (MODE 0) and the numeric
// accumulation (MODE 1: table order, or ascending with c.sort). The warps share a
// column without a barrier (walk_entries): by rounds of B entries when there are
// enough of them, else by windows of each round's stream, which every warp lays out
// for itself. A CTA-wide scan per chunk of B entries (block_walk) waited on
// four barriers for the few dozen entries of such a column and took 29 KB of
// shared memory from the tables. Issue of the shared-memory CAS and add bounds
// the walk now. Measured against block_walk, protein product of 100k columns
// (int64 indices, float): numeric 1173 -> 1091 us (8192 slots), 504 -> 390 us
// (4096), 168 -> 149 us (2048), symbolic 163 -> 125 us (4096); a stage of R-MAT
// scale 15 split in four: numeric 155 -> 135 us (16384), 91 -> 79 us (8192),
// symbolic 95 -> 79 us (16384).
// Registers: 64 let one CTA of 1024 threads run; the symbolic tables up to 8192 slots
// leave room for half as many threads again at 40 (protein symbolic 330 -> 270 us at 8192,
// 125 -> 102 us at 4096), which slows the numeric pass (8192 slots 1090 -> 1107 us, 16384
// slots 139 -> 163 us per stage of the R-MAT).
template <class V> constexpr int mid_smem(int T, int threads, int mode) {
    return T * (4 + (mode == 1 ? (int)sizeof(V) : 0)) + threads * (8 + (mode == 1 ? (int)sizeof(V) : 0));
}

template <class I, class V, int T, int MODE>
__global__ void __maxnreg__(MODE == 0 && T <= 8192 ? 40 : 64) k_mid(GemmArgs<I, V> ga, TierCommon c, I *out_rows, V *out_vals) {
    constexpr int LOG2T = Log2<T>::v;
    extern __shared__ __align__(16) unsigned char smem[];
    V *vals = reinterpret_cast<V *>(smem);
    uint32_t *keys = reinterpret_cast<uint32_t *>(smem + (MODE == 1 ? sizeof(V) * T : 0));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int64_t *off = reinterpret_cast<int64_t *>(keys + T) + warp * 32;
    V *sbv = reinterpret_cast<V *>(reinterpret_cast<int64_t *>(keys + T) + nw * 32) + warp * 32;
    __shared__ SortShared ss;
    __shared__ int s_it, s_red[33];
    const ProbDev<I, V> *pd = ga.probs;
    const I *bp = pd->bp;
    const int lo = c.list_off[c.tier], hi = c.list_off[c.tier + 1];
    uint4 *k4 = reinterpret_cast<uint4 *>(keys);
    for (int s = threadIdx.x; s < T / 4; s += blockDim.x) k4[s] = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
    if (MODE == 1)
        for (int s = threadIdx.x; s < T; s += blockDim.x) vals[s] = V(0);
    // thread 0 reserves the next column when it starts one
    int ahead = 0;
    if (threadIdx.x == 0) ahead = atomicAdd(c.next_col, 1);
    for (;;) {
        if (threadIdx.x == 0) {
            s_it = lo + ahead;
            ahead = atomicAdd(c.next_col, 1);
        }
        __syncthreads();   // the table is clean, too
        const int it = s_it;
        if (it >= hi) break;
        const int64_t g = c.list[it];
        const int64_t b0 = (int64_t)__ldg(&bp[g]);
        const int nb = (int)((int64_t)__ldg(&bp[g + 1]) - b0);
        int64_t out0 = 0;
        int want = 0;
        if (MODE == 1) {
            out0 = c.colptr[g] - c.out_base;
            want = (int)(c.colptr[g + 1] - c.colptr[g]);
        }
        int mine = 0;
        auto insert = [&](uint32_t r, V x) {
            bool fresh;
            const int h = hash_insert_dbl1(keys, LOG2T, r, c.err, fresh);
            if (MODE == 0) mine += fresh;
            else if (h >= 0) atomic_add_v(&vals[h], x);
        };
        const bool rounds = nb >= 64 * nw;
        walk_entries<MODE>(pd, ga.k0, ga.k1, b0, nb, rounds ? warp : 0, rounds ? nw : 1, rounds ? 0 : warp,
                           rounds ? 1 : nw, off, sbv, insert);
        if (MODE == 0) {
            mine = warp_sum(mine);
            if (lane == 0) s_red[warp] = mine;
            __syncthreads();
            if (warp == 0) {
                const int v = warp_sum(lane < nw ? s_red[lane] : 0);
                if (lane == 0) c.cnt[g] = v;
            }
            for (int s = threadIdx.x; s < T / 4; s += blockDim.x) k4[s] = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
            __syncthreads();   // before thread 0 names the next column
            continue;
        }
        __syncthreads();
        if (c.sort) {
            sorted_emit<true>(keys, vals, T, want, &ss, c.err, out_rows + out0, out_vals + out0);
            continue;
        }
        // a warp owns a run of slots: count, one barrier, write and clear
        const int per = (T + nw - 1) / nw;
        const int slo = min(T, warp * per), shi = min(T, slo + per);
        int n = 0;
        for (int s = slo + lane; s < shi; s += 32) n += keys[s] != kEmpty;
        n = warp_sum(n);
        int o = warp_offset(n, s_red, warp, nw, lane);
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
                keys[s] = kEmpty;
                vals[s] = V(0);
            }
            o += __popc(bal);
        }
        if (warp == nw - 1 && lane == 0 && o != want) atomicOr(c.err, kErrCount);
        __syncthreads();
    }
}

// Masked backward of light columns (columns of G of at most T / 2 entries),
// one warp each: for every product A(i, k) B(k, j) with G(i, j) stored,
//   dA(i, k) += G(i, j) B(k, j),  dB(k, j) += A(i, k) G(i, j).
// G(:, j) is looked up in a warp-private table. The products are walked as one
// stream with four windows of loads in flight; a window's lanes in one segment
// (one B entry) add up their parts of dB in registers, so dB takes one global
// add per segment and window, and dA's adds go to consecutive entries. Walking
// one segment after another with an add per product for both took 377 us for
// configuration 5 (12.8 M products), now 189 us (and dB is closer to its 64-bit value: 4.8e-8 against 6.5e-8).
template <class I, class V, int T>
__global__ void __launch_bounds__(256) k_bwd_light(GradArgs<I, V> a, TierCommon c) {
    constexpr int LOG2T = Log2<T>::v;
    constexpr int U = 4;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    V *gv = reinterpret_cast<V *>(smem) + warp * T;
    uint32_t *keys = reinterpret_cast<uint32_t *>(smem + sizeof(V) * 8 * T) + warp * T;
    unsigned char *segs = smem + (size_t)8 * T * (4 + sizeof(V));
    V *s_bv = reinterpret_cast<V *>(segs) + warp * 32;
    int *s_off = reinterpret_cast<int *>(segs + 8 * 32 * sizeof(V)) + warp * 32;
    int *s_e = reinterpret_cast<int *>(segs + 8 * 32 * (sizeof(V) + 4)) + warp * 32;
    const ProbDev<I, V> *pd = a.gemm.probs;
    const I *bp = pd->bp, *bi = pd->bi, *ap = pd->ap, *ai = pd->ai;
    const V *bv = pd->bv, *av = pd->av;
    V *dA = a.dA, *dB = a.dB;
    const int64_t k0 = a.gemm.k0, k1 = a.gemm.k1;
    const unsigned below = (1u << lane) - 1u, upto = 0xffffffffu >> (31 - lane);
    const unsigned above = ~upto;
    const int lo = c.list_off[c.tier], hi = c.list_off[c.tier + 1];
    uint4 *k4 = reinterpret_cast<uint4 *>(keys);
    for (int s = lane; s < T / 4; s += 32) k4[s] = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
    __syncwarp();
    for (int it = lo + blockIdx.x * 8 + warp; it < hi; it += gridDim.x * 8) {
        const int64_t g = c.list[it];
        int64_t gb, ge;
        g_range(a, g, gb, ge);
        const int64_t b0 = (int64_t)__ldg(&bp[g]);
        const int nb = (int)((int64_t)__ldg(&bp[g + 1]) - b0);
        for (int64_t q = gb + lane; q < ge; q += 32) {
            const int h = hash_insert_dbl1(keys, LOG2T, (uint32_t)a.grows[q], c.err);
            if (h >= 0) gv[h] = a.gvals[q];
        }
        __syncwarp();
        for (int base = 0; base < nb; base += 32) {
            int beg = 0, len = 0;
            V bval = V(0);
            if (base + lane < nb) {
                const int64_t k = (int64_t)__ldg(&bi[b0 + base + lane]);
                if (k >= k0 && k < k1) {   // an index outside [0, k) is skipped, as everywhere
                    const int64_t s = (int64_t)__ldg(&ap[k]);
                    beg = (int)s;
                    len = (int)((int64_t)__ldg(&ap[k + 1]) - s);
                }
                bval = __ldg(&bv[b0 + base + lane]);
            }
            const int incl = warp_incl_scan(len);
            const int excl = incl - len;
            const int tot = __shfl_sync(SPG_FULL, incl, 31);
            const unsigned nzm = __ballot_sync(SPG_FULL, len > 0);
            if (len > 0) {
                const int rank = __popc(nzm & below);
                s_off[rank] = beg - excl;
                s_bv[rank] = bval;
                s_e[rank] = base + lane;
            }
            __syncwarp();
            int before = -1;   // segments started before the window, minus one
            for (int w = 0; w < tot; w += 32 * U) {
                uint32_t r[U];
                V x[U];
                int q[U], sl[U];
                unsigned M[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int p = w + 32 * u + lane;
                    const unsigned d = (unsigned)(excl - (w + 32 * u));
                    M[u] = __reduce_or_sync(SPG_FULL, len > 0 && d < 32u ? 1u << d : 0u);
                    sl[u] = before + __popc(M[u] & upto);
                    before += __popc(M[u]);
                    q[u] = -1;
                    if (p < tot) {
                        q[u] = s_off[sl[u]] + p;
                        r[u] = (uint32_t)__ldg(&ai[q[u]]);
                        x[u] = __ldg(&av[q[u]]);
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (w + 32 * u >= tot) break;   // the same for the warp
                    V part = V(0);
                    if (q[u] >= 0) {
                        // the table holds G(:, j): empty slot first means not stored
                        const uint32_t key = r[u];
                        uint32_t h = hash_slot(key, LOG2T);
                        const uint32_t step = ((key * 0x85EBCA6Bu) >> (32 - LOG2T)) | 1u;
                        uint32_t cur = keys[h];
                        for (int probe = 0; probe < T && cur != key && cur != kEmpty; ++probe) {
                            h = (h + step) & (T - 1);
                            cur = keys[h];
                        }
                        if (cur == key) {
                            const V gval = gv[h];
                            atomic_add_v(&dA[q[u]], mul_v(gval, s_bv[sl[u]]));
                            part = mul_v(x[u], gval);
                        }
                    }
                    __syncwarp();
                    // sum over the lanes of the segment, into its first lane
                    const unsigned later = M[u] & above;
                    const int end = later ? __ffs(later) - 1 : 32;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const V y = shfl_bits(part, lane + o < 32 ? lane + o : lane);
                        if (lane + o < end) part = add_v(part, y);
                    }
                    if (q[u] >= 0 && (lane == 0 || ((M[u] >> lane) & 1u))) atomic_add_v(&dB[b0 + s_e[sl[u]]], part);
                }
            }
            __syncwarp();   // the segments are read: the next round may replace them
        }
        for (int s = lane; s < T / 4; s += 32) k4[s] = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
        __syncwarp();
    }
}

}  // namespace spg
