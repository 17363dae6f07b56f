// Algorithm 1 (Section 3.3) on block indices, in closed form.  With equal, aligned query and key blocks the
// window and power-of-two terms depend on the block distance d = i - j only, the sink term on j, and
// causality on j <= i.  With w = max(W, 1) (distance 0 always passes: 0 & -1 == 0) the ascending list of
// query block i is three runs without duplicates:
//   sink    j = 0, 1, ...       the sink blocks outside the window:    j < S, j <= i - w
//   power   j = i - 2^k         k descending, where no other run has it: 2^k >= w, i - 2^k >= S
//   window  j = max(0, i - w + 1) .. i
// so the number of entries, the entry at a position and the number of entries of all rows before a row are
// each a few integer operations: rows need no walk and the CSR no scan.
#pragma once

#include <stdint.h>

namespace pa {

struct LayoutRow {
    int64_t i, w0;            // the query block, first block of its window
    int32_t sinks, powers;    // lengths of the first two runs
    int32_t kmax;             // exponent of the first power entry
    int64_t n;                // entries of the row
};

__host__ __device__ inline int64_t layout_clamp(int64_t x, int64_t hi) { return x < 0 ? 0 : x < hi ? x : hi; }

// floor(log2 x), x >= 1
__host__ __device__ inline int layout_log2(int64_t x)
{
#ifdef __CUDA_ARCH__
    return 63 - __clzll(x);
#else
    return 63 - __builtin_clzll((unsigned long long)x);
#endif
}

// i >= 0, W >= 0, S >= 0.  `power` false drops the power-of-two run: the sliding-window pattern (local window
// plus sink blocks, Section 3.2 / Section 4.1 "Baseline").
__host__ __device__ inline LayoutRow layout_row(int64_t i, int32_t W, int32_t S, bool power = true)
{
    const int64_t w = W > 1 ? W : 1;
    LayoutRow r;
    r.i = i;
    r.w0 = i - w + 1 > 0 ? i - w + 1 : 0;
    r.sinks = (int32_t)layout_clamp(i - w + 1, S);
    const int k0 = w > 1 ? layout_log2(w - 1) + 1 : 0;  // first k with 2^k >= w
    r.kmax = power && i - S >= 1 ? layout_log2(i - S) : -1;
    r.powers = r.kmax >= k0 ? r.kmax - k0 + 1 : 0;
    r.n = (i - r.w0 + 1) + r.sinks + r.powers;
    return r;
}

// The entry at position pos of the row (0 <= pos < n).
__host__ __device__ inline int64_t layout_entry(const LayoutRow &r, int64_t pos)
{
    if (pos < r.sinks) return pos;
    pos -= r.sinks;
    if (pos < r.powers) return r.i - ((int64_t)1 << (r.kmax - (int)pos));
    return r.w0 + pos - r.powers;
}

// Entries of rows 0 .. n - 1.
__host__ __device__ inline int64_t layout_rows_before(int64_t n, int32_t W, int32_t S, bool power = true)
{
    const int64_t w = W > 1 ? W : 1;
    const int64_t m = n - w > 0 ? n - w : 0;  // rows that reach beyond their window
    const int64_t a = n < w ? n : w, b = m < S ? m : S;
    int64_t total = a * (a + 1) / 2 + m * w + b * (b + 1) / 2 + (m - b) * S;
    if (power)
        for (int64_t pw = w > 1 ? (int64_t)2 << layout_log2(w - 1) : 1; pw + S < n; pw *= 2) total += n - pw - S;
    return total;
}

// Tile layouts: the mask's block holds r tiles of the attention kernel.  Algorithm 1's window, power and sink
// terms see the blocks only, so every listed block j < i contributes its r tiles; its causal term cuts the
// diagonal block i, the last one listed, down to the tiles i r .. t.  Entry e of tile row t is tile e % r of
// the block at position e / r.  r = 1 is the block layout itself.
__host__ __device__ inline int64_t tile_row_entries(const LayoutRow &row, int64_t t, int32_t r)
{
    return r * (row.n - 1) + (t - row.i * r + 1);
}
__host__ __device__ inline int64_t tile_rows_before(int64_t t, int32_t r, int32_t W, int32_t S, bool power = true)
{
    const int64_t i = t / r, rest = t - i * r;
    const int64_t before = r * (r * (layout_rows_before(i, W, S, power) - i)) + i * ((int64_t)r * (r + 1) / 2);
    return before + rest * r * (layout_row(i, W, S, power).n - 1) + rest * (rest + 1) / 2;
}

}  // namespace pa
