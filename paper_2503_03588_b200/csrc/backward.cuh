// Shared between the backward pass's two translation units: the argument block of its kernels and
// the entry of the tensor-core (tcgen05) kernels.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace pa {

constexpr int kBwdBlk = 64;       // tokens per block
constexpr int kBwdMaxChunk = 32;  // query blocks per chunk of the dK / dV kernels, at most
constexpr size_t kBwdStatusBytes = 256;  // status block at the head of the workspace ([0] error code, [1] detail)
// Words of the status block: items drawn by the tcgen05 kernels; 1 once the preparation is over.
constexpr int kBwdDqCounter = 16, kBwdDkvCounter = 24, kBwdPrepared = 32;

struct BackwardArgs {
    const __nv_bfloat16 *q, *k, *v, *o, *d_o;
    const float *lse;          // [batch, Hq, N]
    const int32_t *row_ptr, *col_idx;
    int32_t *status;           // [0] error code, [1] detail (bounded waits of the tensor-core kernels)
    float *delta;              // [batch, Hq, N]
    int32_t *col_ptr;          // [nqb + 1]: extents of the transposed lists
    int32_t *row_idx;          // [nnz]: query blocks that list each key block, ascending
    int32_t chunk;             // query blocks per chunk of a column, at most
    float *dq, *dk, *dv;       // fp32, contiguous [batch, N, H, D]
    int64_t q_sb, q_ss, q_sh, k_sb, k_ss, k_sh, v_sb, v_ss, v_sh, o_sb, o_ss, o_sh;
    int64_t N;
    int32_t nqb, batch, Hq, Hkv, G;
    int32_t npairs;            // head pairs per KV group: ceil(G / 2)
    int32_t early;             // one wave of work: the next kernel may start beside this one's last blocks
    int32_t prezero;           // the preparation clears all of dK and dV (else a kernel of its own clears what needs it)
    float scale, scale_log2;
    long long wait_cycles;     // limit of every barrier wait of the tensor-core kernels
};

// A chunk of a key block's list: the unit of work of the dK / dV kernels.  Column j owns the chunk slots
// [col_ptr[j] / chunk + j, col_ptr[j + 1] / chunk + j + 1): at least ceil(count / chunk) of them for any
// count, and known from col_ptr alone.  A column of several chunks is cut into equal parts; a slot beyond
// its chunks is empty.
struct BackwardChunk {
    int32_t j, e0, e1;  // key block, extent in row_idx (empty: e0 == e1)
    int32_t parts;      // chunks of the column
};
__device__ __forceinline__ BackwardChunk backward_chunk_at(const BackwardArgs &a, int32_t c)
{
    BackwardChunk r = {0, 0, 0, 0};
    int32_t lo = 0, hi = a.nqb;  // last column whose slots start at or before c
    while (hi - lo > 1) {
        const int32_t mid = (lo + hi) >> 1;
        if (a.col_ptr[mid] / a.chunk + mid <= c) lo = mid;
        else hi = mid;
    }
    const int32_t p0 = a.col_ptr[lo], cnt = a.col_ptr[lo + 1] - p0;
    const int32_t parts = (cnt + a.chunk - 1) / a.chunk, part = c - (p0 / a.chunk + lo);
    r.j = lo;
    r.parts = parts;
    if (part < parts) {
        r.e0 = p0 + (int32_t)((int64_t)cnt * part / parts);
        r.e1 = p0 + (int32_t)((int64_t)cnt * (part + 1) / parts);
    }
    return r;
}

// The same found by a whole warp: 32 columns compared at a time, two rounds of loads up to 1024 key blocks where the
// halving above takes ten.
__device__ __forceinline__ BackwardChunk backward_chunk_by_warp(const BackwardArgs &a, int32_t c, int lane)
{
    int32_t lo = 0, hi = a.nqb, step, p = 0, p_next = 0, at;
    do {
        step = (hi - lo + 31) / 32;
        const int32_t x = lo + lane * step;
        p = x < hi ? a.col_ptr[x] : 0;
        p_next = x < hi ? a.col_ptr[x + 1] : 0;
        // (column lo starts at or before c, so the lanes that do are the first ones)
        at = __popc(__ballot_sync(0xffffffffu, x < hi && p / a.chunk + x <= c)) - 1;
        lo += at * step;
        if (lo + step < hi) hi = lo + step;
    } while (step > 1);
    const int32_t p0 = __shfl_sync(0xffffffffu, p, at), cnt = __shfl_sync(0xffffffffu, p_next, at) - p0;
    const int32_t parts = (cnt + a.chunk - 1) / a.chunk, part = c - (p0 / a.chunk + lo);
    BackwardChunk r = {lo, 0, 0, parts};
    if (part < parts) {
        r.e0 = p0 + (int32_t)((int64_t)cnt * part / parts);
        r.e1 = p0 + (int32_t)((int64_t)cnt * (part + 1) / parts);
    }
    return r;
}

// dQ, dK and dV on tcgen05 (delta and the transposed lists are already in the workspace).
pa_status launch_backward_sm100(const BackwardArgs &a, const pa_prefill_params *p, int64_t nnz, int device, int sms,
                                cudaStream_t st);

}  // namespace pa
