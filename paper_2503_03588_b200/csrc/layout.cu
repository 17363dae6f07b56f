// pa_layout_size / pa_build_layout: the block-sparse CSR of Algorithm 1 (Section 3.3).
#include <vector>

#include "common.cuh"
#include "layout_rule.cuh"

namespace pa {

// One warp per row writes row_ptr[t] and the row's entries, both in closed form: one launch, nothing to scan,
// coalesced stores.  (128K tokens: 2.8 us in a graph; count, one-block scan and fill with a thread per row were
// three launches and 8.2 us, and the host summed the size row by row twice, 80 us.)
constexpr int kLayoutThreads = 128;

__global__ void __launch_bounds__(kLayoutThreads) layout_kernel(int32_t n_rows, int32_t r, int32_t W, int32_t S, bool power,
                                                                int32_t *row_ptr, int32_t *col_idx)
{
    const int64_t t = (int64_t)blockIdx.x * (kLayoutThreads / 32) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    pdl_launch_next();
    const int64_t start = tile_rows_before(t, r, W, S, power);
    pdl_wait();  // (nothing of global memory is touched before this)
    if (t > n_rows) return;
    if (lane == 0) row_ptr[t] = (int32_t)start;
    if (t == n_rows) return;
    const LayoutRow row = layout_row(t / r, W, S, power);
    const int64_t n = tile_row_entries(row, t, r);
    for (int64_t e = lane; e < n; e += 32) {
        const int64_t pos = r == 1 ? e : e / r;
        col_idx[start + e] = (int32_t)(layout_entry(row, pos) * r + (e - pos * r));
    }
}

static pa_status check_layout_args(int64_t seq_len, int32_t block, int32_t W, int32_t S)
{
    if (seq_len < 1) return fail(PA_ERR_INVALID_ARG, "seq_len must be >= 1 (got %lld)", (long long)seq_len);
    if (block < 1) return fail(PA_ERR_INVALID_ARG, "block must be >= 1 (got %d)", block);
    if (W < 0 || S < 0) return fail(PA_ERR_INVALID_ARG, "window_blocks and sink_blocks must be >= 0");
    return PA_OK;
}

// Sizes and arrays of a layout listed in tiles, r = block / tile of them per block (r = 1: in blocks).
static pa_status layout_size(int64_t seq_len, int32_t tile, int32_t r, int32_t W, int32_t S, bool power, int32_t *n_rows,
                             int64_t *nnz)
{
    if (!n_rows || !nnz) return fail(PA_ERR_INVALID_ARG, "the row count and nnz pointers must be non-null");
    const int64_t rows = (seq_len + tile - 1) / tile;
    if (rows >= INT32_MAX) return fail(PA_ERR_SHAPE, "%lld rows do not fit in int32", (long long)rows);
    // (a window or a sink of more blocks than there are rows lists no more than that many: no overflow below)
    const int32_t cap = (int32_t)(rows / r + 2);
    const int64_t total = tile_rows_before(rows, r, W < cap ? W : cap, S < cap ? S : cap, power);
    if (total > INT32_MAX) return fail(PA_ERR_SHAPE, "nnz %lld does not fit in int32", (long long)total);
    *n_rows = (int32_t)rows;
    *nnz = total;
    return PA_OK;
}

static pa_status check_window(int32_t W)
{
    if (W < 1)
        return fail(PA_ERR_INVALID_ARG, "a sliding-window layout needs window_blocks >= 1 (the diagonal block)");
    return PA_OK;
}

static pa_status check_tile(int32_t block, int32_t tile)
{
    if (tile < 1) return fail(PA_ERR_INVALID_ARG, "tile must be >= 1 (got %d)", tile);
    if (block % tile != 0) return fail(PA_ERR_SHAPE, "block %d is not a multiple of tile %d", block, tile);
    return PA_OK;
}

static pa_status build_layout(int64_t seq_len, int32_t tile, int32_t r, int32_t W, int32_t S, bool power, int32_t *row_ptr,
                              int32_t *col_idx, int64_t col_capacity, void *stream)
{
    int32_t rows = 0;
    int64_t nnz = 0;
    if (pa_status s = layout_size(seq_len, tile, r, W, S, power, &rows, &nnz)) return s;
    if (!row_ptr || !col_idx) return fail(PA_ERR_INVALID_ARG, "row_ptr and col_idx must be non-null");
    if (col_capacity < nnz)
        return fail(PA_ERR_LAYOUT, "col_capacity %lld < nnz %lld", (long long)col_capacity, (long long)nnz);
    constexpr int kRowsPerBlock = kLayoutThreads / 32;
    PA_CUDA_OK(launch_pdl(layout_kernel, dim3((unsigned)(((int64_t)rows + kRowsPerBlock) / kRowsPerBlock)), kLayoutThreads, 0,
                          static_cast<cudaStream_t>(stream), rows, r, W, S, power, row_ptr, col_idx));
    return PA_OK;
}

}  // namespace pa

extern "C" pa_status pa_layout_size(int64_t seq_len, int32_t block, int32_t window_blocks,
                                    int32_t sink_blocks, int32_t *n_qblocks, int64_t *nnz)
{
    using namespace pa;
    clear_error();
    if (pa_status s = check_layout_args(seq_len, block, window_blocks, sink_blocks)) return s;
    return layout_size(seq_len, block, 1, window_blocks, sink_blocks, true, n_qblocks, nnz);
}

extern "C" pa_status pa_build_layout(int64_t seq_len, int32_t block, int32_t window_blocks,
                                     int32_t sink_blocks, int32_t *row_ptr, int32_t *col_idx,
                                     int64_t col_capacity, void *stream)
{
    using namespace pa;
    clear_error();
    if (pa_status s = check_layout_args(seq_len, block, window_blocks, sink_blocks)) return s;
    return build_layout(seq_len, block, 1, window_blocks, sink_blocks, true, row_ptr, col_idx, col_capacity, stream);
}

extern "C" pa_status pa_window_layout_size(int64_t seq_len, int32_t block, int32_t window_blocks,
                                           int32_t sink_blocks, int32_t *n_qblocks, int64_t *nnz)
{
    using namespace pa;
    clear_error();
    if (pa_status s = check_layout_args(seq_len, block, window_blocks, sink_blocks)) return s;
    if (pa_status s = check_window(window_blocks)) return s;
    return layout_size(seq_len, block, 1, window_blocks, sink_blocks, false, n_qblocks, nnz);
}

extern "C" pa_status pa_build_window_layout(int64_t seq_len, int32_t block, int32_t window_blocks,
                                            int32_t sink_blocks, int32_t *row_ptr, int32_t *col_idx,
                                            int64_t col_capacity, void *stream)
{
    using namespace pa;
    clear_error();
    if (pa_status s = check_layout_args(seq_len, block, window_blocks, sink_blocks)) return s;
    if (pa_status s = check_window(window_blocks)) return s;
    return build_layout(seq_len, block, 1, window_blocks, sink_blocks, false, row_ptr, col_idx, col_capacity, stream);
}

extern "C" pa_status pa_reach_counts(const int32_t *row_ptr, const int32_t *col_idx, int32_t n_blocks,
                                     int32_t start, int32_t max_steps, int64_t *counts)
{
    using namespace pa;
    clear_error();
    if (!row_ptr || !col_idx || !counts) return fail(PA_ERR_INVALID_ARG, "row_ptr, col_idx and counts must be non-null");
    if (n_blocks < 1 || start < 0 || start >= n_blocks || max_steps < 1)
        return fail(PA_ERR_INVALID_ARG, "need n_blocks >= 1, 0 <= start < n_blocks, max_steps >= 1");
    // Breadth-first search from `start` over the edges block -> listed key block, level by level.
    std::vector<int32_t> depth((size_t)n_blocks, -1), frontier{start}, next;
    depth[(size_t)start] = 0;
    int64_t reached = 1;
    for (int32_t k = 1; k <= max_steps; ++k) {
        next.clear();
        for (int32_t u : frontier) {
            const int32_t lo = row_ptr[u], hi = row_ptr[u + 1];
            if (lo < 0 || hi < lo) return fail(PA_ERR_LAYOUT, "row %d has a negative extent", u);
            for (int32_t e = lo; e < hi; ++e) {
                const int32_t v = col_idx[e];
                if (v < 0 || v >= n_blocks) return fail(PA_ERR_LAYOUT, "row %d lists block %d outside [0, %d)", u, v, n_blocks);
                if (depth[(size_t)v] < 0) {
                    depth[(size_t)v] = k;
                    next.push_back(v);
                    ++reached;
                }
            }
        }
        counts[k - 1] = reached;
        frontier.swap(next);
    }
    return PA_OK;
}

extern "C" pa_status pa_tile_layout_size(int64_t seq_len, int32_t block, int32_t window_blocks,
                                         int32_t sink_blocks, int32_t tile, int32_t *n_qtiles, int64_t *nnz)
{
    using namespace pa;
    clear_error();
    if (pa_status s = check_layout_args(seq_len, block, window_blocks, sink_blocks)) return s;
    if (pa_status s = check_tile(block, tile)) return s;
    return layout_size(seq_len, tile, block / tile, window_blocks, sink_blocks, true, n_qtiles, nnz);
}

extern "C" pa_status pa_build_tile_layout(int64_t seq_len, int32_t block, int32_t window_blocks,
                                          int32_t sink_blocks, int32_t tile, int32_t *row_ptr,
                                          int32_t *col_idx, int64_t col_capacity, void *stream)
{
    using namespace pa;
    clear_error();
    if (pa_status s = check_layout_args(seq_len, block, window_blocks, sink_blocks)) return s;
    if (pa_status s = check_tile(block, tile)) return s;
    return build_layout(seq_len, tile, block / tile, window_blocks, sink_blocks, true, row_ptr, col_idx, col_capacity, stream);
}
