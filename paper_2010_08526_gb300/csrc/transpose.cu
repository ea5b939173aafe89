// spgemm_transpose: the CSC of A^T (equivalently the CSR of A) on the device.
// A^T serves A A^T (Sec. V's BELLA workload) and the row-by-row batching the
// paper mentions for square inputs (Sec. IV-B): the row batches of C = A B
// are the column batches of C^T = B^T A^T.
//
//   1. count[i] = entries in row i of A      (one atomic per entry)
//   2. colptr of A^T = exclusive scan of count
//   3. every entry (i, j, v) of A goes to a slot of column i of A^T, taken
//      with an atomic cursor: row index j, value v.
// Values are moved as raw 4- or 8-byte words. Rows inside an output column
// come in an unspecified order (as every output of the library).
#include <algorithm>
#include <string>

#include "../../include/spgemm.h"
#include "plan.h"
#include "util.h"

namespace spg {

// rows outside [0, m) are skipped and flagged (corrupt input)
template <class I>
__global__ void k_t_count(const I *rowidx, int64_t nnz, int64_t m, unsigned long long *count, int *err) {
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nnz; q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = (int64_t)rowidx[q];
        if (i < 0 || i >= m) { atomicOr(err, 1); continue; }
        atomicAdd(&count[i], 1ull);
    }
}

// A warp takes `window` consecutive entries, four per lane at a time: the columns of
// the first and of the last one by a search in colptr (half of the lanes each), and every
// entry's column between these two. A warp per column left 30 lanes idle on columns of
// two entries, the shape of a k-mer matrix (the call on 800,018 entries 0.34 ms, now 0.10); a
// whole search per entry cost more than it saved on long columns of neighbouring rows, whose
// cursors stay in cache (warp per column / search per entry / now, int32, ms: 2,000,000
// columns of 50 rows 1.90 / 2.65 / 1.61, 4,000,000 of 16 1.66 / 1.98 / 1.15, 100,000 of
// 1000 2.27 / 2.68 / 2.27). 256 entries a warp from kTransLarge on (with 128: 1.74, 1.31,
// 2.37); fewer entries need the warps (4096 columns of 8 rows 0.075 against 0.081).
constexpr int64_t kTransLarge = int64_t(1) << 22;
template <class P, class I, class W>
__global__ void __launch_bounds__(256) k_t_scatter(const P *colptr, const I *rowidx, const W *vals, int64_t ncols,
                                                   int64_t nnz, int64_t m, int window, unsigned long long *cursor,
                                                   I *out_rows, W *out_vals) {
    constexpr int U = 4;
    const int lane = threadIdx.x & 31;
    const int64_t base = (int64_t)colptr[0];
    auto column = [&](int64_t q, int64_t lo, int64_t hi) {   // the last one starting at or before q
        while (lo < hi) {
            const int64_t mid = (lo + hi + 1) >> 1;
            if ((int64_t)__ldg(&colptr[mid]) - base <= q) lo = mid; else hi = mid - 1;
        }
        return lo;
    };
    const int64_t step = (((int64_t)gridDim.x * blockDim.x) >> 5) * window;
    for (int64_t w = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * window; w < nnz; w += step) {
        const int64_t ends = column(lane < 16 ? w : min(w + window, nnz) - 1, 0, ncols - 1);
        const int64_t c0 = __shfl_sync(0xffffffffu, ends, 0), c1 = __shfl_sync(0xffffffffu, ends, 31);
        for (int64_t w1 = w; w1 < min(w + window, nnz); w1 += 32 * U) {
            int64_t i[U], c[U];
            W v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t q = w1 + 32 * u + lane;
                i[u] = q < nnz ? (int64_t)rowidx[q] : -1;
                if (q < nnz) v[u] = vals[q];
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                c[u] = i[u] >= 0 && i[u] < m ? column(w1 + 32 * u + lane, c0, c1) : -1;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (c[u] < 0) continue;
                const unsigned long long pos = atomicAdd(&cursor[i[u]], 1ull);
                out_rows[pos] = (I)c[u];
                out_vals[pos] = v[u];
            }
        }
    }
}

template <class T>
__global__ void k_t_colptr(const int64_t *src, int64_t n, T *dst) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = (T)src[i];
}

template <class P, class I, class W>
static spgemm_status transpose_typed(const spgemm_csc *in, spgemm_csc *out, cudaStream_t st) {
    const int64_t m = in->nrows, n = in->ncols, nnz = in->nnz;
    DevBuf arena, count, scan, part, err;   // parts of one block
    CallScratch scratch(arena, st);
    cudaError_t e = carve<SPGEMM_MEM_DEVICE>(
        arena, {{&count, sizeof(int64_t) * (size_t)(m + 1)}, {&scan, sizeof(int64_t) * (size_t)(m + 1)},
                {&part, sizeof(int64_t) * (size_t)scan_partials_len(m + 1)}, {&err, sizeof(int) * 4}});
    if (e != cudaSuccess) {
        if (e == cudaErrorMemoryAllocation) {
            set_error("transpose: workspace allocation failed");
            return SPGEMM_ERR_OOM;
        }
        return cuda_fail(e, "transpose workspace");
    }
    if ((e = cudaMemsetAsync(count.p, 0, sizeof(int64_t) * (size_t)(m + 1), st)) != cudaSuccess ||
        (e = cudaMemsetAsync(err.p, 0, sizeof(int), st)) != cudaSuccess)
        return cuda_fail(e, "cudaMemsetAsync");
    const unsigned eb = (unsigned)std::max<int64_t>(1, std::min<int64_t>((nnz + 255) / 256, 1 << 20));
    const int window = nnz >= kTransLarge ? 256 : 128;
    const unsigned wb = (unsigned)std::max<int64_t>(1, std::min<int64_t>((nnz + 8 * window - 1) / (8 * window), 1 << 20));
    const unsigned mb = (unsigned)std::max<int64_t>(1, std::min<int64_t>((m + 256) / 256, 1 << 20));
    // entry q of the input is rowidx[q - colptr[0]] (the pointers address
    // the first entry), as everywhere in the library
    if (nnz > 0)
        k_t_count<I><<<eb, 256, 0, st>>>((const I *)in->rowidx, nnz, m, count.as<unsigned long long>(), err.as<int>());
    if ((e = exclusive_scan_i64(count.as<int64_t>(), m, scan.as<int64_t>(), part.as<int64_t>(), 1, st)) != cudaSuccess)
        return cuda_fail(e, "scan");
    if (out->ptr_type == SPGEMM_I64) k_t_colptr<int64_t><<<mb, 256, 0, st>>>(scan.as<int64_t>(), m + 1, (int64_t *)out->colptr);
    else k_t_colptr<int32_t><<<mb, 256, 0, st>>>(scan.as<int64_t>(), m + 1, (int32_t *)out->colptr);
    if (nnz > 0)
        k_t_scatter<P, I, W><<<wb, 256, 0, st>>>((const P *)in->colptr, (const I *)in->rowidx, (const W *)in->vals, n,
                                                 nnz, m, window, scan.as<unsigned long long>(), (I *)out->rowidx, (W *)out->vals);
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "transpose kernels");
    // the workspace is freed on return: wait for the kernels that use it
    int herr = 0;
    if ((e = cudaMemcpyAsync(&herr, err.p, sizeof(int), cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
        (e = cudaStreamSynchronize(st)) != cudaSuccess)
        return cuda_fail(e, "cudaStreamSynchronize");
    if (herr) { set_error("transpose: a row index lies outside [0, nrows)"); return SPGEMM_ERR_INVALID; }
    return SPGEMM_OK;
}

}  // namespace spg

using namespace spg;

extern "C" spgemm_status spgemm_transpose(const spgemm_csc *in, spgemm_csc *out, cudaStream_t stream) {
    if (!in || !out) { set_error("NULL argument"); return SPGEMM_ERR_INVALID; }
    if (in->nrows < 0 || in->ncols < 0 || in->nnz < 0 || in->nrows >= 0x7fffffffLL || in->ncols >= 0x7fffffffLL) {
        set_error("transpose: bad shape (dimensions must be < 2^31-1)"); return SPGEMM_ERR_INVALID;
    }
    if (!in->colptr || (in->nnz > 0 && (!in->rowidx || !in->vals))) {
        set_error("transpose: NULL input array"); return SPGEMM_ERR_INVALID;
    }
    if (out->nrows != in->ncols || out->ncols != in->nrows || out->nnz != in->nnz ||
        out->idx_type != in->idx_type || out->val_type != in->val_type || !out->colptr ||
        (in->nnz > 0 && (!out->rowidx || !out->vals)) ||
        (out->ptr_type != SPGEMM_I32 && out->ptr_type != SPGEMM_I64) ||
        (in->ptr_type != SPGEMM_I32 && in->ptr_type != SPGEMM_I64)) {
        set_error("transpose: out must be ncols x nrows with the input's nnz, index and value types");
        return SPGEMM_ERR_INVALID;
    }
    if (out->ptr_type == SPGEMM_I32 && in->nnz >= 0x7fffffffLL) {
        set_error("transpose: nnz does not fit a 32-bit colptr"); return SPGEMM_ERR_INDEX_OVERFLOW;
    }
    const bool p64 = in->ptr_type == SPGEMM_I64, i64 = in->idx_type == SPGEMM_I64;
    const bool w8 = in->val_type != SPGEMM_F32;
#define TR(P, I, W) return transpose_typed<P, I, W>(in, out, stream)
    if (p64) {
        if (i64) { if (w8) TR(int64_t, int64_t, uint64_t); else TR(int64_t, int64_t, uint32_t); }
        else { if (w8) TR(int64_t, int32_t, uint64_t); else TR(int64_t, int32_t, uint32_t); }
    } else {
        if (i64) { if (w8) TR(int32_t, int64_t, uint64_t); else TR(int32_t, int64_t, uint32_t); }
        else { if (w8) TR(int32_t, int32_t, uint64_t); else TR(int32_t, int32_t, uint32_t); }
    }
#undef TR
}
