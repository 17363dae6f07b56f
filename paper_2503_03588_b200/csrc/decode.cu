// pa_decode / pa_decode_paged: one query token per sequence against its KV cache under the
// PowerAttention row of its position (Section 4.1: same pattern in prefilling and decoding;
// Eq. (1) for the row).  The cache is either one contiguous [batch, max_len, Hkv, D] array or a
// pool of 64-token pages reached through a block table.
//
// Two paths.  Rows with at most 32 window, power-of-two and sink candidates (every PowerAttention
// row with the default window up to millions of tokens) take one launch: decode_cluster_kernel where they are few (a
// thread-block cluster per (sequence, KV head)), else decode_row_kernel (a CTA per row), described at those kernels.
// Longer rows take the split-K pair below.
//
// Split-K: one CTA per (sequence, KV head, chunk) where a chunk is one 64-key block of the
// row's block list.  Each CTA reads its K and V block with coalesced 16-byte loads and computes
// the logits of all query heads of the group, a chunk-local softmax and the unnormalised partial
// output on the warp-level tensor-core MMA.  The chunk partials (o[D], m, l) are then merged with
// the log-sum-exp rule by a second kernel, launched with programmatic dependent launch so that
// its start-up overlaps the first kernel's tail; it waits for the partials with griddepcontrol.wait.
#include <cuda.h>
#include <cuda_bf16.h>
#include <math.h>
#include <stdlib.h>

#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "layout_rule.cuh"
#include "sm100_ptx.cuh"
#include "tensor_map.cuh"

namespace pa {

constexpr int kDecBlock = 64;     // keys per block (the only supported block size)
constexpr int kDecThreads = 128;  // threads per CTA of the partial kernel
constexpr int kMaxGroup = 8;      // query heads per KV head supported by the decode kernels
constexpr size_t kDecStatusBytes = 256;  // status block at the start of the workspace

struct DecodeArgs {
    const __nv_bfloat16 *q, *k, *v;
    const int32_t *lens;
    const int32_t *table;  // paged cache: [batch, table_stride] page numbers; null: contiguous cache
    float *partial;        // [batch, Hq, chunks, D + 2]
    int32_t *status;       // [0] error code, [1] detail
    int32_t clear_status;  // the kernel clears the error code itself
    void *o;
    float *lse;
    // Element strides.  Contiguous cache: batch, token, head.  Paged: page, token in page, head.
    int64_t k_sb, k_ss, k_sh, v_sb, v_ss, v_sh;
    int64_t max_len;
    int32_t batch, Hq, Hkv, G, W, S, chunks, o_is_f32;
    int32_t stages;        // (row and cluster kernels) shared-memory stages of this launch
    int32_t R;             // (row and cluster kernels) chunks per row
    int32_t fixed_chunks;  // (combine kernel) > 0: every row has this many partials
    int64_t items;         // (row kernel) rows of the call x R
    int32_t table_stride, n_pages;
    float scale_log2;  // softmax_scale * log2(e)
    long long wait_cycles;  // (row and cluster kernels) limit of every barrier wait, in clock cycles
};

// Where key block j of sequence b starts: (index along the batch / page axis, first token).  A
// page number outside the pool is clamped (the result is then undefined but nothing faults).
__device__ __forceinline__ void block_origin(const DecodeArgs &a, int b, int32_t j, int64_t &outer, int64_t &tok0)
{
    if (a.table) {
        int32_t page = a.table[(int64_t)b * a.table_stride + j];
        page = page < 0 ? 0 : (page >= a.n_pages ? a.n_pages - 1 : page);
        outer = page;
        tok0 = 0;
    } else {
        outer = b;
        tok0 = (int64_t)j * kDecBlock;
    }
}

// Loads that stay where they are written, ahead of the work that hides them.  (Not the read-only kind: decode_row_kernel
// may start while the kernel that writes what it reads still runs.)
__device__ __forceinline__ uint4 ld16(const void *p)
{
    uint4 r;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
                 : "l"(p)
                 : "memory");
    return r;
}
__device__ __forceinline__ uint32_t ld4(const void *p)
{
    uint32_t r;
    asm volatile("ld.global.u32 %0, [%1];\n" : "=r"(r) : "l"(p) : "memory");
    return r;
}

// D(16x8, fp32) += A(16x16, bf16, row-major) * B(16x8, bf16, column-major), one warp.
__device__ __forceinline__ void mma_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Attention of one 64-key block for all query heads of a KV group.
//
// Logits: each of the four warps takes 16 keys; the query heads of the group are the M rows of
// the 16 x 8 x 16 MMA (rows beyond the group are zero), so one pass over K serves every head.
// K, V and Q are read straight from global memory with 16-byte loads, all issued before the
// first use.  A thread's 16-byte piece holds eight consecutive features of one row; the dot
// product does not care in which order features are paired, so the pieces are fed to the MMA
// fragments as they come (Q and K use the same pairing).  The logits go through shared memory
// once so that every warp sees the whole 64-key row and the block's softmax uses one maximum.
// Output: each warp owns 32 of the features and runs P V over all 64 keys for them (two rows of
// V are interleaved with byte permutes to form the B fragments), so no cross-warp merge is needed.
template <int D>
__global__ void __launch_bounds__(kDecThreads) decode_block_kernel(const DecodeArgs a)
{
    // Let the combine kernel's CTAs be scheduled as soon as SM resources free up.
    pdl_launch_next();
    constexpr int NJ = D / 32;  // 16-byte pieces per thread and row for Q and K
    __shared__ float sS[kMaxGroup][kDecBlock + 8];  // base-2 logits of the block

    const int chunk = blockIdx.x, hk = blockIdx.y, b = blockIdx.z;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int g = lane >> 2, t = lane & 3;
    const int G = a.G;
    if (chunk == 0 && hk == 0 && b == 0 && tid == 0) a.status[0] = 0;  // no bounded waits on this path

    const int64_t len = a.lens[b];
    const bool valid = len >= 1 && len <= a.max_len;
    const int64_t p = len - 1;
    const int32_t row = valid ? (int32_t)(p / kDecBlock) : 0;  // max_len / 64 fits in 31 bits (host check)
    const LayoutRow list = layout_row(row, a.W, a.S);
    if (!valid || chunk >= list.n) return;
    const int32_t jblk = (int32_t)layout_entry(list, chunk);  // this CTA's key block

    {
        const int n_keys = jblk == row ? (int)(p % kDecBlock) + 1 : kDecBlock;
        const int base = wid * 16;            // first key of this warp's logit tile
        const int vchunk = (g & 3) + 4 * wid;  // this thread's 8-feature piece of V rows
        const bool pv_warp = 4 * wid < D / 8;  // warps that own output features

        // ---- loads (keys at or beyond n_keys do not exist: zeros instead of a read)
        int64_t outer, tok0;
        block_origin(a, b, jblk, outer, tok0);
        const __nv_bfloat16 *kb = a.k + outer * a.k_sb + tok0 * a.k_ss + hk * a.k_sh;
        const __nv_bfloat16 *vb = a.v + outer * a.v_sb + tok0 * a.v_ss + hk * a.v_sh;
        const uint4 zero4 = make_uint4(0, 0, 0, 0);
        uint4 kr[2][NJ], vr[4][4], qr[NJ];
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
            const int key = base + nt * 8 + g;
#pragma unroll
            for (int j = 0; j < NJ; ++j)
                kr[nt][j] = key < n_keys ? ld16(kb + key * a.k_ss + 8 * (4 * j + t)) : zero4;
        }
        const __nv_bfloat16 *qb = a.q + ((int64_t)b * a.Hq + (int64_t)hk * G + g) * D;
#pragma unroll
        for (int j = 0; j < NJ; ++j) qr[j] = g < G ? ld16(qb + 8 * (4 * j + t)) : zero4;
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
#pragma unroll
            for (int kx = 0; kx < 4; ++kx) {
                const int key = 16 * ks + 2 * t + (kx & 1) + (kx >> 1) * 8;
                vr[ks][kx] = (pv_warp && key < n_keys) ? ld16(vb + key * a.v_ss + 8 * vchunk) : zero4;
            }

        // ---- S = Q K^T: rows = heads, columns = the warp's 16 keys (two 8-key tiles)
        float sc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                mma_bf16(sc[nt], qr[j].x, 0u, qr[j].y, 0u, kr[nt][j].x, kr[nt][j].y);
                mma_bf16(sc[nt], qr[j].z, 0u, qr[j].w, 0u, kr[nt][j].z, kr[nt][j].w);
            }
        }
        // This thread holds head g, keys base + 8 nt + 2 t + {0, 1}: to shared memory in the
        // base-2 domain (s * scale * log2(e)); keys that do not exist become -inf.
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
            const int key = base + nt * 8 + 2 * t;
            float2 v2;
            v2.x = key < n_keys ? sc[nt][0] * a.scale_log2 : -INFINITY;
            v2.y = key + 1 < n_keys ? sc[nt][1] * a.scale_log2 : -INFINITY;
            *reinterpret_cast<float2 *>(&sS[g][key]) = v2;
        }
        __syncthreads();

        // ---- block softmax: thread (g, t) takes keys 16 ks + {2t, 2t+1, 2t+8, 2t+9}, ks = 0..3
        // (exactly the positions of its P fragments); the four t lanes cover the row.
        float2 sv[4][2];
        float mrow = -INFINITY;
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                sv[ks][hh] = *reinterpret_cast<const float2 *>(&sS[g][16 * ks + 8 * hh + 2 * t]);
                mrow = fmaxf(mrow, fmaxf(sv[ks][hh].x, sv[ks][hh].y));
            }
        mrow = fmaxf(mrow, __shfl_xor_sync(0xffffffffu, mrow, 1));
        mrow = fmaxf(mrow, __shfl_xor_sync(0xffffffffu, mrow, 2));  // finite: key 0 of the block exists
        uint32_t pa[4][2];
        float lrow = 0.f;
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                const float p0 = ptx::ex2(sv[ks][hh].x - mrow), p1 = ptx::ex2(sv[ks][hh].y - mrow);
                lrow += p0 + p1;
                const __nv_bfloat162 h2 = __floats2bfloat162_rn(p0, p1);
                pa[ks][hh] = *reinterpret_cast<const uint32_t *>(&h2);
            }
        lrow += __shfl_xor_sync(0xffffffffu, lrow, 1);
        lrow += __shfl_xor_sync(0xffffffffu, lrow, 2);
        if (wid == 0 && t == 0 && g < G) {
            float *dst = a.partial + (((int64_t)b * a.Hq + hk * G + g) * a.chunks + chunk) * (D + 2);
            dst[D] = mrow;      // base-2 maximum of the block
            dst[D + 1] = lrow;  // sum of 2^(s2 - m)
        }

        // ---- O = P V for this warp's 32 features.  Lanes g and g + 4 read the same 16-byte piece
        // and take its low / high half: feature tile e covers features 8 vchunk(n) + e + 4 (n >> 2)
        // for n = 0..7.
        if (pv_warp) {
            const bool hi = (g >> 2) != 0;
            float acc[4][4];
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[e][0] = acc[e][1] = acc[e][2] = acc[e][3] = 0.f;
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
                uint32_t w0[2], w1[2], w2[2], w3[2];  // the two 32-bit words this lane uses, per key
                w0[0] = hi ? vr[ks][0].z : vr[ks][0].x; w0[1] = hi ? vr[ks][0].w : vr[ks][0].y;
                w1[0] = hi ? vr[ks][1].z : vr[ks][1].x; w1[1] = hi ? vr[ks][1].w : vr[ks][1].y;
                w2[0] = hi ? vr[ks][2].z : vr[ks][2].x; w2[1] = hi ? vr[ks][2].w : vr[ks][2].y;
                w3[0] = hi ? vr[ks][3].z : vr[ks][3].x; w3[1] = hi ? vr[ks][3].w : vr[ks][3].y;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t sel = (e & 1) ? 0x7632u : 0x5410u;
                    const uint32_t b0 = __byte_perm(w0[e >> 1], w1[e >> 1], sel);
                    const uint32_t b1 = __byte_perm(w2[e >> 1], w3[e >> 1], sel);
                    mma_bf16(acc[e], pa[ks][0], 0u, pa[ks][1], 0u, b0, b1);
                }
            }
            // acc[e][x]: head g, column n = 2t + x of the tile -> feature below.
            if (g < G) {
                float *dst = a.partial + (((int64_t)b * a.Hq + hk * G + g) * a.chunks + chunk) * (D + 2);
#pragma unroll
                for (int e = 0; e < 4; ++e)
#pragma unroll
                    for (int x = 0; x < 2; ++x) {
                        const int nn = 2 * t + x;
                        dst[8 * ((nn & 3) + 4 * wid) + e + 4 * (nn >> 2)] = acc[e][x];
                    }
            }
        }
    }
}

// Log-sum-exp merge of the chunk partials of one (sequence, query head):
//   m = max m_c,  l = sum l_c 2^(m_c - m),  o = sum o_c 2^(m_c - m) / l,  LSE = (m + log2 l) ln 2.
template <int D>
__global__ void __launch_bounds__(D) decode_combine_kernel(const DecodeArgs a)
{
    __shared__ float s_red[D / 32];
    const int h = blockIdx.x, b = blockIdx.y, d = threadIdx.x;
    // The partial kernel's writes are visible only after this wait (and so are the lengths: the kernel before it
    // in the stream may have written them, and nothing has waited for that one yet).
    pdl_wait();
    pdl_launch_next();
    const int64_t len = a.lens[b];
    const bool valid = len >= 1 && len <= a.max_len;
    int n = 0;
    if (valid) n = a.fixed_chunks > 0 ? a.fixed_chunks : (int)layout_row((len - 1) / kDecBlock, a.W, a.S).n;
    const float *src = a.partial + (((int64_t)b * a.Hq + h) * a.chunks) * (D + 2);
    // Global maximum: the chunks are spread over the threads (independent loads), then reduced.
    float m = -INFINITY;
    for (int c = d; c < n; c += D) m = fmaxf(m, src[c * (D + 2) + D]);
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((d & 31) == 0) s_red[d >> 5] = m;
    __syncthreads();
    m = s_red[0];
#pragma unroll
    for (int w = 1; w < D / 32; ++w) m = fmaxf(m, s_red[w]);
    // Weighted sums; the loop is unrolled so that the loads of several chunks are in flight.
    float l = 0.f, acc = 0.f;
#pragma unroll 8
    for (int c = 0; c < n; ++c) {
        const float w = exp2f(src[c * (D + 2) + D] - m);
        l += src[c * (D + 2) + D + 1] * w;
        acc += src[c * (D + 2) + d] * w;
    }
    const float out = n > 0 ? acc / l : 0.f;
    const int64_t oi = ((int64_t)b * a.Hq + h) * D + d;
    if (a.o_is_f32)
        reinterpret_cast<float *>(a.o)[oi] = out;
    else
        reinterpret_cast<__nv_bfloat16 *>(a.o)[oi] = __float2bfloat16_rn(out);
    if (d == 0) a.lse[(int64_t)b * a.Hq + h] = n > 0 ? (m + log2f(l)) * 0.6931471805599453f : -INFINITY;
}

// ------------------------------------------------------------------------------------------
// The row kernel: attention of (sequence, KV head) rows whose block set fits one warp's lanes.
//
// A row's key blocks are dealt round-robin to R chunks; a work item is one chunk of one row.
// Inside a CTA:
//   warp 4      producer: one elected lane walks the items' blocks and fetches each K block and
//               each V block with TMA box loads (64 keys x 64 features, 128-byte swizzle) into a
//               ring of shared-memory stages; K and V complete on separate mbarriers, so the
//               logits start as soon as K has landed.  The ring runs on across items: while the
//               consumers finish one item the next one's blocks are already on their way.
//   warps 0-3   consumers: warp w owns keys 16 w .. 16 w + 15 of every block.  Logits on the
//               warp-level MMA with the group's query heads as the M rows (K fragments by
//               ldmatrix), online softmax in registers (running maximum, sum and output kept across
//               blocks), O += P V for all D features (V fragments by transposing ldmatrix).  No
//               block-wide barrier inside the loop: a warp only waits for a stage to fill and
//               says when it has finished with it.  At the end of an item the four warps merge
//               their partial results through shared memory with the log-sum-exp rule, each
//               warp a quarter of the features.
// A persistent grid of two CTAs per SM strides over the items.  With one chunk per row (the default) O and LSE are
// written straight from the registers; with more (kParts, only under PA_DECODE_CLUSTER) each item's (o, m, l) goes to
// the workspace and decode_combine_kernel merges a row's R chunks (second launch, programmatic dependent launch).
// Every mbarrier wait is bounded; one that runs out records PA_ERR_TIMEOUT in the status block
// and the CTA runs to its end without hanging.
// ------------------------------------------------------------------------------------------
constexpr int kRowConsumers = 4;                     // consumer warps
constexpr int kRowThreads = 32 * (kRowConsumers + 1);
constexpr int kRowMaxStages = 6;                     // shared-memory stages (key blocks in flight) per CTA
constexpr int kRowMaxCluster = 8;                    // portable cluster size limit
constexpr int kRowMaxSmem = 227 * 1024;              // dynamic shared memory a CTA may ask for
constexpr long long kRowWaitCycles = 2000000000ll;   // default limit of a barrier wait: ~1 s

template <int D>
struct RowSmem {
    static constexpr uint32_t kSub = kDecBlock * 128;        // 64 keys x 64 features
    static constexpr uint32_t kTile = kSub * (D / 64);       // one K or V block
    static constexpr uint32_t kStage = 2 * kTile;            // K + V of one key block
    // Hand-over area of the end-of-item merge: per warp and head, the tiles the warp does not own
    // (three quarters of the D features) and its running maximum and sum.
    static constexpr uint32_t kPartRow = D - D / 4 + 2;
    static constexpr uint32_t kPart = kRowConsumers * kMaxGroup * kPartRow * 4;
    static constexpr uint32_t kBars = 3 * kRowMaxStages * 8 + 16;
    static constexpr size_t bytes(int stages) { return 1024 + (size_t)stages * kStage + kPart + kBars; }
};

// The row's block set, one candidate per lane (the order does not matter for Eq. (1), so the set
// is not sorted): window distances 0 .. w-1, then the power-of-two distances >= w that do not
// land on a sink block, then the sink blocks outside the window.  Returns this lane's key block
// or -1.  The host takes the cluster and row kernels only when window + powers + sinks fit the 32 lanes.
__device__ __forceinline__ int32_t row_block_candidate(int32_t row, int32_t W, int32_t S, int lane)
{
    const int32_t w_eff = W > 1 ? W : 1;
    const int k0 = w_eff <= 1 ? 0 : 32 - __clz(w_eff - 1);  // first k with 2^k >= w_eff
    const int kmax = row >= 1 ? 31 - __clz(row) : -1;       // last k with 2^k <= row
    const int n_pow = kmax >= k0 ? kmax - k0 + 1 : 0;
    int32_t cand = -1;
    if (lane < w_eff) {
        cand = row - lane;  // negative: before the sequence start
    } else if (lane < w_eff + n_pow) {
        const int32_t j = row - (1 << (k0 + lane - w_eff));
        if (j >= S) cand = j;
    } else if (lane < w_eff + n_pow + S) {
        const int32_t j = lane - w_eff - n_pow;
        if (row - j >= w_eff) cand = j;  // also implies j <= row
    }
    return cand;
}

// kParts: rows come in R chunks; else R = 1, known to the compiler (one block of 128 features, 16 rows: 3.6 us against 3.8).
// Registers are what 128 features are short of (168 a thread, two CTAs of five warps per SM).  With the next item's Q in
// registers of its own throughout, and the diagonal block found by its index, this form spilled 104 bytes: 28 / 4 heads, 9000
// tokens, 150 rows 13.0 us, 296 rows 17.0, 512 rows 33.5; so 36 bytes, 11.7, 16.4 and 32.8.
template <int D, bool kParts>
__global__ void __launch_bounds__(kRowThreads, 2) decode_row_kernel(const __grid_constant__ CUtensorMap tmK,
                                                                    const __grid_constant__ CUtensorMap tmV,
                                                                    const DecodeArgs a)
{
    using SM = RowSmem<D>;
    constexpr int DH = D / 64;  // 64-feature (128-byte) sub-tiles per key row
    extern __shared__ uint8_t row_smem_raw[];
    const uint32_t smem_base = (ptx::smem_u32(row_smem_raw) + 1023u) & ~1023u;
    uint8_t *smem = row_smem_raw + (smem_base - ptx::smem_u32(row_smem_raw));
    const int stages = a.stages;
    const uint32_t off_part = (uint32_t)stages * SM::kStage;
    float *part = reinterpret_cast<float *>(smem + off_part);  // [warp][head][kPartRow]
    const uint32_t bars = smem_base + off_part + SM::kPart;
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + off_part + SM::kPart + 3 * kRowMaxStages * 8);
    auto bar_kfull = [&](int s) { return bars + (uint32_t)s * 8u; };
    auto bar_vfull = [&](int s) { return bars + (uint32_t)(kRowMaxStages + s) * 8u; };
    auto bar_empty = [&](int s) { return bars + (uint32_t)(2 * kRowMaxStages + s) * 8u; };

    const int R = kParts ? a.R : 1;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int g = lane >> 2, t = lane & 3;
    const int G = a.G;

    // (item and row counts fit 31 bits; checked on the host)
    const uint32_t n_items = (uint32_t)a.items;
    const uint32_t it0 = blockIdx.x, it_step = gridDim.x;
    // The launch after this one may take the places this one leaves; this one itself has started before the
    // kernel ahead of it was done: up to pdl_wait() nothing of global memory is read or written.
    pdl_launch_next();
    if (tid == 0) {
        for (int s = 0; s < stages; ++s) {
            ptx::mbar_init(bar_kfull(s), 1);
            ptx::mbar_init(bar_vfull(s), 1);
            ptx::mbar_init(bar_empty(s), kRowConsumers);
        }
        *abort_flag = 0;
        ptx::fence_barrier_init();
        ptx::fence_proxy_async_smem();
        ptx::prefetch_tensormap(&tmK);
        ptx::prefetch_tensormap(&tmV);
    }
    __syncthreads();
    pdl_wait();
    const int32_t len_first = it0 < n_items ? a.lens[(it0 / (uint32_t)R) / (uint32_t)a.Hkv] : 0;
    if (a.clear_status && blockIdx.x == 0 && tid == 0) a.status[0] = 0;  // a wait that gives up (much later) sets it

    // Item it -> (row of the call, chunk); a row -> (sequence, KV head).
    struct Item {
        int32_t b, hk, r;        // sequence, KV head, chunk
        int32_t last_keys;       // keys of the diagonal block
        int32_t cand;            // this lane's candidate key block or -1
        int32_t rank;            // its number among the candidates that exist (lane order)
        int32_t page;            // (paged cache) its page
        uint32_t have;           // lanes whose candidate exists
        int32_t n, mine;         // blocks of the row, blocks of this chunk
    };
    auto item_len = [&](uint32_t it) -> int32_t {  // the sequence's cache length (issued early: a global load)
        return it < n_items ? a.lens[(it / (uint32_t)R) / (uint32_t)a.Hkv] : 0;
    };
    auto make_item = [&](uint32_t it, int32_t len32) {
        Item w;
        const int32_t rowid = (int32_t)(it / (uint32_t)R);
        w.r = (int32_t)(it - (uint32_t)rowid * (uint32_t)R);
        w.b = (int32_t)((uint32_t)rowid / (uint32_t)a.Hkv);
        w.hk = rowid - w.b * a.Hkv;
        const int64_t len = len32;
        const bool valid = len >= 1 && len <= a.max_len;
        const int64_t p = len - 1;
        w.last_keys = (int32_t)(p % kDecBlock) + 1;
        w.cand = valid ? row_block_candidate((int32_t)(p / kDecBlock), a.W, a.S, lane) : -1;
        w.page = 0;
        if (a.table && w.cand >= 0) w.page = a.table[(int64_t)w.b * a.table_stride + w.cand];
        w.have = __ballot_sync(0xffffffffu, w.cand >= 0);
        w.rank = __popc(w.have & ((1u << lane) - 1u));
        w.n = __popc(w.have);
        w.mine = w.n > w.r ? (w.n - w.r + R - 1) / R : 0;
        return w;
    };
    // Key block number i of the item: the (r + i R)-th candidate that exists (lane that holds it).
    auto lane_of = [&](const Item &w, int i) {
        const uint32_t hit = __ballot_sync(0xffffffffu, w.cand >= 0 && w.rank == w.r + i * R);
        return (__ffs(hit) - 1) & 31;
    };

    if (wid == kRowConsumers) {
        // ------------------------------------------------------------------ producer
        bool ok = true;
        uint32_t ci = 0;  // blocks issued so far by this CTA (ring position)
        int32_t len_next = len_first;
        for (uint32_t it = it0; it < n_items; it += it_step) {
            const Item w = make_item(it, len_next);
            len_next = item_len(it + it_step);
            for (int i = 0; i < w.mine; ++i, ++ci) {
                const int src = lane_of(w, i);
                const int32_t j = __shfl_sync(0xffffffffu, w.cand, src);
                const int32_t page = __shfl_sync(0xffffffffu, w.page, src);
                if (lane == 0 && ok) {
                    const int s = (int)(ci % (uint32_t)stages);
                    if (ci >= (uint32_t)stages)
                        ok = ptx::mbar_wait_bounded(bar_empty(s), (ci / (uint32_t)stages - 1) & 1, abort_flag, a.status, 1,
                                                    a.wait_cycles, (int)PA_ERR_TIMEOUT);
                    if (ok) {
                        // (a page outside the pool reads as zeros)
                        const int32_t outer = a.table ? page : w.b, tok0 = a.table ? 0 : j * kDecBlock;
                        const uint32_t dst = smem_base + (uint32_t)s * SM::kStage;
                        ptx::mbar_expect_tx(bar_kfull(s), SM::kTile);
#pragma unroll
                        for (int dh = 0; dh < DH; ++dh)
                            ptx::tma_load_4d(dst + dh * SM::kSub, &tmK, bar_kfull(s), dh * 64, tok0, w.hk, outer);
                        ptx::mbar_expect_tx(bar_vfull(s), SM::kTile);
#pragma unroll
                        for (int dh = 0; dh < DH; ++dh)
                            ptx::tma_load_4d(dst + SM::kTile + dh * SM::kSub, &tmV, bar_vfull(s), dh * 64, tok0, w.hk, outer);
                    }
                }
                __syncwarp();
            }
        }
    } else {
        // ------------------------------------------------------------------ consumers
        // ldmatrix row addresses inside a tile.  K (matrices: keys 0-7 / 8-15 of the warp x two
        // 16-byte feature chunks): lane -> key 16 w + 8 (lane / 16) + lane % 8, chunk + (lane / 8) % 2.
        // V (transposed; matrices: two key halves x two feature chunks): key 16 w + 8 ((lane / 8) % 2)
        // + lane % 8, chunk + lane / 16.  A 16-byte chunk c of row `key` sits at c ^ (key % 8).
        const int k_key = 16 * wid + ((lane >> 4) << 3) + (lane & 7), k_ch = (lane >> 3) & 1;
        const int v_key = 16 * wid + (((lane >> 3) & 1) << 3) + (lane & 7), v_ch = lane >> 4;
        // Q fragments: head g is row g of the 16-row A operand (rows 8..15 are zero).  The next item's are requested
        // behind the last product with the current item's, into the same registers.
        uint32_t qa[D / 16][2];
        auto load_q = [&](uint32_t it) {
            const bool in = it < n_items && g < G;
            const int32_t rowid = in ? (int32_t)(it / (uint32_t)R) : 0;  // = b Hkv + hk, and its heads start at rowid G
            const __nv_bfloat16 *qb = a.q + ((int64_t)rowid * G + g) * D;
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) {
                qa[ks][0] = in ? ld4(qb + 16 * ks + 2 * t) : 0u;
                qa[ks][1] = in ? ld4(qb + 16 * ks + 8 + 2 * t) : 0u;
            }
        };
        load_q(it0);
        bool ok = true;
        uint32_t ci = 0;
        int32_t len_next = len_first;
        for (uint32_t it = it0; it < n_items && ok; it += it_step) {
            const Item w = make_item(it, len_next);
            len_next = item_len(it + it_step);
            float m_run = -INFINITY, l_run = 0.f;
            float acc[D / 8][4];
#pragma unroll
            for (int e = 0; e < D / 8; ++e) acc[e][0] = acc[e][1] = acc[e][2] = acc[e][3] = 0.f;
#pragma unroll 1
            for (int i = 0; i < w.mine && ok; ++i, ++ci) {
                const int s = (int)(ci % (uint32_t)stages);
                const uint32_t parity = (ci / (uint32_t)stages) & 1;
                const int n_keys = w.r == 0 && i == 0 ? w.last_keys : kDecBlock;  // (the diagonal block is lane 0's)
                const uint32_t sk = smem_base + (uint32_t)s * SM::kStage, sv = sk + SM::kTile;
                ok = ptx::mbar_wait_bounded(bar_kfull(s), parity, abort_flag, a.status, 2, a.wait_cycles, (int)PA_ERR_TIMEOUT);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                if (16 * wid < n_keys) {  // (else none of this warp's keys exists: the diagonal block's tail)
                    // ---- S = Q K^T: rows = heads, columns = the warp's 16 keys (two 8-key tiles).  K
                    // fragments are requested four feature slices ahead of their MMAs, and each tile
                    // accumulates in two chains (even and odd slices), which halves the dependent-MMA latency.
                    float sc[2][2][4];
#pragma unroll
                    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                        for (int c = 0; c < 2; ++c) sc[nt][c][0] = sc[nt][c][1] = sc[nt][c][2] = sc[nt][c][3] = 0.f;
#pragma unroll
                    for (int kb = 0; kb < D / 16; kb += 4) {
                        uint32_t kf[4][4];
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            const int ch = 2 * (kb + x) + k_ch;
                            ptx::ldmatrix_x4(sk + (uint32_t)(ch >> 3) * SM::kSub + (uint32_t)k_key * 128u +
                                                 (uint32_t)(((ch & 7) ^ (k_key & 7)) << 4),
                                             kf[x][0], kf[x][1], kf[x][2], kf[x][3]);
                        }
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            mma_bf16(sc[0][x & 1], qa[kb + x][0], 0u, qa[kb + x][1], 0u, kf[x][0], kf[x][1]);
                            mma_bf16(sc[1][x & 1], qa[kb + x][0], 0u, qa[kb + x][1], 0u, kf[x][2], kf[x][3]);
                        }
                    }
                    // This thread: head g, keys 16 w + 8 nt + 2 t + {0, 1}; base-2 domain; keys that do
                    // not exist become -inf (a select, so whatever the cache holds there is ignored).
                    const int key0 = 16 * wid + 2 * t;
                    float sx[4];
                    sx[0] = key0 < n_keys ? (sc[0][0][0] + sc[0][1][0]) * a.scale_log2 : -INFINITY;
                    sx[1] = key0 + 1 < n_keys ? (sc[0][0][1] + sc[0][1][1]) * a.scale_log2 : -INFINITY;
                    sx[2] = key0 + 8 < n_keys ? (sc[1][0][0] + sc[1][1][0]) * a.scale_log2 : -INFINITY;
                    sx[3] = key0 + 9 < n_keys ? (sc[1][0][1] + sc[1][1][1]) * a.scale_log2 : -INFINITY;
                    float mx = fmaxf(fmaxf(sx[0], sx[1]), fmaxf(sx[2], sx[3]));
                    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
                    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));  // finite: key 16 w exists
                    const float m_new = fmaxf(m_run, mx);
                    const float alpha = ptx::ex2(m_run - m_new);  // 0 on the warp's first block
                    const float p0 = ptx::ex2(sx[0] - m_new), p1 = ptx::ex2(sx[1] - m_new);
                    const float p2 = ptx::ex2(sx[2] - m_new), p3 = ptx::ex2(sx[3] - m_new);
                    float lsum = (p0 + p1) + (p2 + p3);
                    lsum += __shfl_xor_sync(0xffffffffu, lsum, 1);
                    lsum += __shfl_xor_sync(0xffffffffu, lsum, 2);
                    l_run = l_run * alpha + lsum;
                    m_run = m_new;
                    const uint32_t pa0 = ptx::cvt_bf16x2(p0, p1), pa1 = ptx::cvt_bf16x2(p2, p3);
#pragma unroll
                    for (int e = 0; e < D / 8; ++e) {
                        acc[e][0] *= alpha;
                        acc[e][1] *= alpha;
                    }
                    // V rows of keys that do not exist may hold anything (0 x NaN would poison O):
                    // they are cleared in the fragments.  Only the diagonal block has such rows.
                    uint32_t keep0 = 0xffffffffu, keep1 = 0xffffffffu;
                    if (n_keys < kDecBlock) {
                        keep0 = (key0 < n_keys ? 0x0000ffffu : 0u) | (key0 + 1 < n_keys ? 0xffff0000u : 0u);
                        keep1 = (key0 + 8 < n_keys ? 0x0000ffffu : 0u) | (key0 + 9 < n_keys ? 0xffff0000u : 0u);
                    }
                    ok = ptx::mbar_wait_bounded(bar_vfull(s), parity, abort_flag, a.status, 3, a.wait_cycles,
                                                (int)PA_ERR_TIMEOUT);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    // ---- O = alpha O + P V: rows = heads, 16 keys, all D features (8 per MMA)
#pragma unroll
                    for (int eb = 0; eb < D / 16; eb += 4) {
                        uint32_t vf[4][4];
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            const int ch = 2 * (eb + x) + v_ch;
                            ptx::ldmatrix_x4_trans(sv + (uint32_t)(ch >> 3) * SM::kSub + (uint32_t)v_key * 128u +
                                                       (uint32_t)(((ch & 7) ^ (v_key & 7)) << 4),
                                                   vf[x][0], vf[x][1], vf[x][2], vf[x][3]);
                        }
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            mma_bf16(acc[2 * (eb + x)], pa0, 0u, pa1, 0u, vf[x][0] & keep0, vf[x][1] & keep1);
                            mma_bf16(acc[2 * (eb + x) + 1], pa0, 0u, pa1, 0u, vf[x][2] & keep0, vf[x][3] & keep1);
                        }
                    }
                }
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(bar_empty(s));  // this warp has finished with the stage
            }
            load_q(it + it_step);

            // ---- the four warps' partials are merged with the log-sum-exp rule, each warp taking a
            // quarter of the features (four of the 8-feature tiles): a thread passes on the tiles it
            // does not own and picks up, for the tiles it owns, the very elements its lane holds in
            // the other three warps.
            {
                float *mine_out = part + ((size_t)wid * kMaxGroup + g) * SM::kPartRow;
#pragma unroll
                for (int e = 0; e < D / 8; ++e)
                    if (e / (D / 32) != wid)
                        *reinterpret_cast<float2 *>(mine_out + 8 * (e < wid * (D / 32) ? e : e - D / 32) + 2 * t) =
                            make_float2(acc[e][0], acc[e][1]);
                if (t == 0) {
                    mine_out[SM::kPartRow - 2] = m_run;
                    mine_out[SM::kPartRow - 1] = l_run;
                }
            }
            asm volatile("bar.sync 1, %0;\n" ::"n"(32 * kRowConsumers) : "memory");
            float m = -INFINITY, l = 0.f;
            float fin[D / 32][2];
            {
                float mw[kRowConsumers], lw[kRowConsumers], ww[kRowConsumers];
#pragma unroll
                for (int x = 0; x < kRowConsumers; ++x) {
                    const float *src = part + ((size_t)x * kMaxGroup + g) * SM::kPartRow;
                    mw[x] = x == wid ? m_run : src[SM::kPartRow - 2];
                    lw[x] = x == wid ? l_run : src[SM::kPartRow - 1];
                    m = fmaxf(m, mw[x]);
                }
#pragma unroll
                for (int x = 0; x < kRowConsumers; ++x) {
                    ww[x] = mw[x] != -INFINITY ? ptx::ex2(mw[x] - m) : 0.f;
                    l = fmaf(lw[x], ww[x], l);
                }
#pragma unroll
                for (int y = 0; y < D / 32; ++y) {
                    fin[y][0] = fin[y][1] = 0.f;
#pragma unroll
                    for (int x = 0; x < kRowConsumers; ++x) {
                        // warp x keeps this warp's tile y at slot (tile index among the tiles x does not own)
                        const int e = wid * (D / 32) + y;
                        float2 v2;
                        if (x == wid) {
                            v2 = make_float2(0.f, 0.f);  // (own tiles: taken from registers below)
                        } else {
                            const float *src = part + ((size_t)x * kMaxGroup + g) * SM::kPartRow;
                            v2 = *reinterpret_cast<const float2 *>(src + 8 * (e < x * (D / 32) ? e : e - D / 32) + 2 * t);
                        }
                        fin[y][0] = fmaf(v2.x, ww[x], fin[y][0]);
                        fin[y][1] = fmaf(v2.y, ww[x], fin[y][1]);
                    }
                }
                // own tiles out of the accumulators (the tile index depends on the warp: a uniform switch)
#pragma unroll
                for (int e = 0; e < D / 8; ++e)
                    if (e / (D / 32) == wid) {
                        fin[e % (D / 32)][0] = fmaf(acc[e][0], ww[wid], fin[e % (D / 32)][0]);
                        fin[e % (D / 32)][1] = fmaf(acc[e][1], ww[wid], fin[e % (D / 32)][1]);
                    }
            }
            // Thread (g, t) of warp w now holds head g, features (D / 4) w + 8 y + 2 t + {0, 1} of the result.
            {
                const int64_t head = ((int64_t)w.b * a.Hq + (int64_t)w.hk * G + g);
                const int f0 = wid * (D / 4) + 2 * t;
                if (g < G) {
                    if (kParts) {
                        float *dst = a.partial + (head * R + w.r) * (D + 2);
#pragma unroll
                        for (int y = 0; y < D / 32; ++y)
                            *reinterpret_cast<float2 *>(dst + f0 + 8 * y) = make_float2(fin[y][0], fin[y][1]);
                        if (wid == 0 && t == 0) {
                            dst[D] = m;
                            dst[D + 1] = l;
                        }
                    } else {
                        const float inv = w.n > 0 ? 1.0f / l : 0.f;
                        if (a.o_is_f32) {
                            float *dst = reinterpret_cast<float *>(a.o) + head * D + f0;
#pragma unroll
                            for (int y = 0; y < D / 32; ++y)
                                *reinterpret_cast<float2 *>(dst + 8 * y) = make_float2(fin[y][0] * inv, fin[y][1] * inv);
                        } else {
                            __nv_bfloat16 *dst = reinterpret_cast<__nv_bfloat16 *>(a.o) + head * D + f0;
#pragma unroll
                            for (int y = 0; y < D / 32; ++y)
                                *reinterpret_cast<uint32_t *>(dst + 8 * y) = ptx::cvt_bf16x2(fin[y][0] * inv, fin[y][1] * inv);
                        }
                        if (wid == 0 && t == 0)
                            a.lse[head] = w.n > 0 ? (m + log2f(l)) * 0.6931471805599453f : -INFINITY;
                    }
                }
            }
            // The hand-over area is written again only after every warp has read it.
            asm volatile("bar.sync 1, %0;\n" ::"n"(32 * kRowConsumers) : "memory");
        }
    }

    __syncthreads();
    if (*abort_flag && tid == 0) {
        // A wait gave up: leave copies that may still be in flight a bounded time to land
        // before the CTA's shared memory is handed to another CTA.
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000ll) {
        }
    }
}

// ------------------------------------------------------------------------------------------
// The cluster kernel: the same rows in calls of so few that latency is all that counts.
//
// A row's key blocks are dealt round-robin to the R CTAs of a thread-block cluster; a CTA works on two blocks at a time,
// eight warps on 16 keys each for the logits.  The warps exchange their maxima and their weights through shared
// memory, and each takes D / 8 features of O += P V over all keys of the two blocks: what a warp holds at the end is
// the CTA's result for its features, with nothing to merge inside the CTA.  It is pushed to the CTA that merges the
// head (CTA h % R; asynchronous stores that count their bytes on a barrier of the receiving CTA, so that this CTA waits for
// its parts and for nothing else).
// Bound by that chain of latencies.  Measured in a graph, G = 7, head_dim 128, 4000 tokens, against this split done by
// decode_row_kernel (keys kept apart by warp up to the end, the warps' outputs merged in shared memory, then all parts
// behind a barrier of the cluster): 4 rows 3.8 us (5.2), 32 rows 5.0 (6.8), 74 rows 6.8 (8.0), 148 rows 9.2 (10.0).
// ------------------------------------------------------------------------------------------
constexpr int kClusterThreads = 256;
constexpr int kClusterWarps = kClusterThreads / 32;

template <int D>
struct ClusterSmem {
    static constexpr uint32_t kSub = kDecBlock * 128;   // 64 keys x 64 features
    static constexpr uint32_t kTile = kSub * (D / 64);  // one K or V block
    static constexpr uint32_t kStage = 2 * kTile;       // K + V of one key block
    // Weights of a head: 128 keys, bf16; the pad spreads the banks.  Rows 8 .. 15: what that rounding left of them.
    static constexpr uint32_t kPPitch = 2 * kDecBlock * 2 + 16;
    static constexpr uint32_t kMax = 2 * kMaxGroup * kPPitch;  // (behind the weights) [head][warp] maxima
    static constexpr uint32_t kSum = kMax + kMaxGroup * kClusterWarps * 4;  // [head][warp] sums
    // What the row's CTAs send to the CTA that merges a head: per sending CTA and head slot, o[D], m, l.
    // R senders x ceil(8 / R) heads of an owner is at most 14 entries (R = 7).
    static constexpr uint32_t kRecv = kSum + kMaxGroup * kClusterWarps * 4;
    static constexpr uint32_t kRecvRow = (D + 2) * 4;
    static constexpr uint32_t kBars = kRecv + ((14 * kRecvRow + 15) & ~15u);
    static constexpr uint32_t kRest = kBars + (2 * kRowMaxStages + 2) * 8;
    static constexpr size_t bytes(int stages) { return 1024 + (size_t)stages * kStage + kRest; }
};

template <int D>
__global__ void __launch_bounds__(kClusterThreads, 2)
decode_cluster_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, const DecodeArgs a)
{
    using SM = ClusterSmem<D>;
    constexpr int DH = D / 64;            // 64-feature (128-byte) sub-tiles per key row
    constexpr int NT = D / 64;            // 8-feature tiles of O per warp
    extern __shared__ uint8_t row_smem_raw[];
    const uint32_t smem_base = (ptx::smem_u32(row_smem_raw) + 1023u) & ~1023u;
    const int stages = a.stages;
    const uint32_t rest = smem_base + (uint32_t)stages * SM::kStage, bars = rest + SM::kBars;
    volatile int *abort_flag = reinterpret_cast<volatile int *>(row_smem_raw + (bars - ptx::smem_u32(row_smem_raw)) +
                                                                (2 * kRowMaxStages + 1) * 8);
    auto bar_kfull = [&](int s) { return bars + (uint32_t)s * 8u; };
    auto bar_vfull = [&](int s) { return bars + (uint32_t)(kRowMaxStages + s) * 8u; };
    const uint32_t bar_recv = bars + 2 * kRowMaxStages * 8;
    auto wait_bar = [&](uint32_t b_, uint32_t parity, int code) {
        return ptx::mbar_wait_bounded(b_, parity, abort_flag, a.status, code, a.wait_cycles, (int)PA_ERR_TIMEOUT);
    };

    const int R = a.R, G = a.G;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int g = lane >> 2, t = lane & 3;
    const uint32_t rowid = blockIdx.x / (uint32_t)R;  // = b Hkv + hk
    const int r = (int)(blockIdx.x - rowid * (uint32_t)R);
    const uint32_t b = rowid / (uint32_t)a.Hkv, hk = rowid - b * (uint32_t)a.Hkv;
    const uint32_t inv_R = (65536u + (uint32_t)R - 1) / (uint32_t)R;  // x / R = x inv_R >> 16 for x < 32
    // Heads r, r + R, ... are merged here.
    const int heads_here = G > r ? (G - r + R - 1) / R : 0, heads_per_owner = (kMaxGroup + R - 1) / R;

    // The launch after this one may take the places this one leaves; this one itself has started before the
    // kernel ahead of it was done: up to pdl_wait() nothing of global memory is read or written.
    pdl_launch_next();
    if (tid == 0) {
        for (int s = 0; s < stages; ++s) {
            ptx::mbar_init(bar_kfull(s), 1);
            ptx::mbar_init(bar_vfull(s), 1);
        }
        ptx::mbar_init(bar_recv, 1);
        *abort_flag = 0;
        ptx::fence_barrier_init();
        ptx::fence_proxy_async_smem();
        ptx::mbar_expect_tx(bar_recv, (uint32_t)(heads_here * R) * SM::kRecvRow);
        ptx::prefetch_tensormap(&tmK);
        ptx::prefetch_tensormap(&tmV);
    }
    __syncthreads();
    // A peer's shared memory may be written only once the peer has started and set its barrier up.  Each CTA says so here
    // and asks for the others just before it pushes its parts, which hides the answer's way behind the loads.
    ptx::cluster_arrive();
    pdl_wait();
    const int32_t len = a.lens[b];
    if (a.clear_status && blockIdx.x == 0 && tid == 0) a.status[0] = 0;  // a wait that gives up (much later) sets it
    // Q fragments: head g is row g of the 16-row A operand (rows 8..15 are zero).
    uint32_t qa[D / 16][2];
    {
        const bool in = g < G;
        const __nv_bfloat16 *qb = a.q + ((int64_t)rowid * G + (in ? g : 0)) * D;
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) {
            qa[ks][0] = in ? ld4(qb + 16 * ks + 2 * t) : 0u;
            qa[ks][1] = in ? ld4(qb + 16 * ks + 8 + 2 * t) : 0u;
        }
    }

    // The row's block set, one candidate per lane; block number i of this CTA is the (r + i R)-th that exists.  The diagonal
    // block, lane 0's, is block 0 of CTA 0.
    const bool valid = len >= 1 && (int64_t)len <= a.max_len;
    const int32_t row = valid ? (len - 1) / kDecBlock : 0;
    const int32_t cand = valid ? row_block_candidate(row, a.W, a.S, lane) : -1;
    const uint32_t have = __ballot_sync(0xffffffffu, cand >= 0);
    const int n = __popc(have), mine = n > r ? (int)(((uint32_t)(n - r + R - 1) * inv_R) >> 16) : 0;
    const uint32_t rank = (uint32_t)__popc(have & ((1u << lane) - 1u)), quot = (rank * inv_R) >> 16;
    const int my_block = cand >= 0 && (int)(rank - quot * (uint32_t)R) == r ? (int)quot : -1;
    // Warp 0: each lane fetches the block that it found.  (A page outside the pool reads as zeros.)
    int32_t outer = (int32_t)b, tok0 = cand * kDecBlock;
    if (wid == 0 && a.table && my_block >= 0) {
        outer = a.table[(int64_t)b * a.table_stride + cand];
        tok0 = 0;
    }
    auto fetch = [&](int first, int end) {
        if (my_block < first || my_block >= end) return;
        const int s = my_block % stages;
        const uint32_t dst = smem_base + (uint32_t)s * SM::kStage;
        ptx::mbar_expect_tx(bar_kfull(s), SM::kTile);
#pragma unroll
        for (int dh = 0; dh < DH; ++dh) ptx::tma_load_4d(dst + dh * SM::kSub, &tmK, bar_kfull(s), dh * 64, tok0, (int)hk, outer);
        ptx::mbar_expect_tx(bar_vfull(s), SM::kTile);
#pragma unroll
        for (int dh = 0; dh < DH; ++dh)
            ptx::tma_load_4d(dst + SM::kTile + dh * SM::kSub, &tmV, bar_vfull(s), dh * 64, tok0, (int)hk, outer);
    };
    if (wid == 0) {
        fetch(0, stages);
        __syncwarp();
    }

    // ldmatrix row addresses inside a tile.  K (matrices: keys 0-7 / 8-15 of the warp x two 16-byte feature chunks): lane
    // -> key 16 (w % 4) + 8 (lane / 16) + lane % 8, chunk + (lane / 8) % 2.  V (transposed; matrices: two key halves x two
    // feature chunks, or with 64 features four key halves): key 8 (..) + lane % 8.  A 16-byte chunk c of row `key` sits
    // at c ^ (key % 8).
    const int k_key = 16 * (wid & 3) + ((lane >> 4) << 3) + (lane & 7), k_ch = (lane >> 3) & 1;
    const uint32_t p_mine = rest + (uint32_t)g * SM::kPPitch + (uint32_t)(16 * wid + 2 * t) * 2u;
    const uint32_t stat_mine = (uint32_t)(g * kClusterWarps + wid) * 4u, stat_row = (uint32_t)(g * kClusterWarps) * 4u;
    // P as the A operand by ldmatrix: 16 rows (the heads, and their weights' remainders) x 16 keys.
    const uint32_t p_frag = rest + (uint32_t)(lane & 15) * SM::kPPitch + (uint32_t)(lane >> 4) * 16u;
    const int per = stages > 1 ? 2 : 1;  // blocks at a time
    float m_run = -INFINITY, l_run = 0.f;  // of head g: the CTA's maximum, this warp's sum
    float acc[NT][4];
#pragma unroll
    for (int e = 0; e < NT; ++e) acc[e][0] = acc[e][1] = acc[e][2] = acc[e][3] = 0.f;
#pragma unroll 1
    for (int i0 = 0; i0 < mine; i0 += per) {
        const int blocks = min(per, mine - i0);
        const int i = i0 + (wid >> 2);  // this warp's block
        const int n_keys = (wid >> 2) >= blocks ? 0 : r == 0 && i == 0 ? (len - 1) % kDecBlock + 1 : kDecBlock;
        float sx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
        float mx = -INFINITY;
        if (16 * (wid & 3) < n_keys) {
            const int s = i % stages;
            wait_bar(bar_kfull(s), (uint32_t)(i / stages) & 1, 2);
            __syncwarp();
            // ---- S = Q K^T: rows = heads, columns = the warp's 16 keys (two 8-key tiles), two chains of MMAs each.
            const uint32_t sk = smem_base + (uint32_t)s * SM::kStage;
            float sc[2][2][4];
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int x = 0; x < 2; ++x) sc[nt][x][0] = sc[nt][x][1] = sc[nt][x][2] = sc[nt][x][3] = 0.f;
#pragma unroll
            for (int kb = 0; kb < D / 16; kb += 4) {
                uint32_t kf[4][4];
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const int ch = 2 * (kb + x) + k_ch;
                    ptx::ldmatrix_x4(sk + (uint32_t)(ch >> 3) * SM::kSub + (uint32_t)k_key * 128u +
                                         (uint32_t)(((ch & 7) ^ (k_key & 7)) << 4),
                                     kf[x][0], kf[x][1], kf[x][2], kf[x][3]);
                }
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    mma_bf16(sc[0][x & 1], qa[kb + x][0], 0u, qa[kb + x][1], 0u, kf[x][0], kf[x][1]);
                    mma_bf16(sc[1][x & 1], qa[kb + x][0], 0u, qa[kb + x][1], 0u, kf[x][2], kf[x][3]);
                }
            }
            // This thread: head g, keys 8 nt + 2 t + {0, 1} of the warp's 16; base-2 domain; keys that do not exist
            // become -inf (a select, so whatever the cache holds there is ignored).
            const int key0 = 16 * (wid & 3) + 2 * t;
            sx[0] = key0 < n_keys ? (sc[0][0][0] + sc[0][1][0]) * a.scale_log2 : -INFINITY;
            sx[1] = key0 + 1 < n_keys ? (sc[0][0][1] + sc[0][1][1]) * a.scale_log2 : -INFINITY;
            sx[2] = key0 + 8 < n_keys ? (sc[1][0][0] + sc[1][1][0]) * a.scale_log2 : -INFINITY;
            sx[3] = key0 + 9 < n_keys ? (sc[1][0][1] + sc[1][1][1]) * a.scale_log2 : -INFINITY;
            mx = fmaxf(fmaxf(sx[0], sx[1]), fmaxf(sx[2], sx[3]));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        }
        if (t == 0) ptx::st_shared(rest + SM::kMax + stat_mine, __float_as_uint(mx));
        __syncthreads();
        float m_new = m_run;
        {
            float mw[kClusterWarps];
            ptx::ld_shared_v4(rest + SM::kMax + stat_row, mw[0], mw[1], mw[2], mw[3]);
            ptx::ld_shared_v4(rest + SM::kMax + stat_row + 16, mw[4], mw[5], mw[6], mw[7]);
#pragma unroll
            for (int x = 0; x < kClusterWarps; ++x) m_new = fmaxf(m_new, mw[x]);  // finite: a listed block has a key
        }
        const float alpha = ptx::ex2(m_run - m_new);  // 0 at first
        const float p0 = ptx::ex2(sx[0] - m_new), p1 = ptx::ex2(sx[1] - m_new);
        const float p2 = ptx::ex2(sx[2] - m_new), p3 = ptx::ex2(sx[3] - m_new);
        // A weight is split in two bf16 parts, of which the MMA's rows 8 .. 15, otherwise empty, take the second.  All keys
        // share one maximum here (in decode_row_kernel each warp's largest weight is 1, exact in bf16), and with the first
        // part alone the error against 64 bits was 1.2 to 2.5 times that kernel's (8 x 4 rows, 4000 tokens, relative: 1.0e-3
        // there, 1.3e-3 with one part, 1.9e-6 with two, for 0 to 0.2 us a call).
        const uint32_t h01 = ptx::cvt_bf16x2(p0, p1), h23 = ptx::cvt_bf16x2(p2, p3);
        ptx::st_shared(p_mine, h01);
        ptx::st_shared(p_mine + 16, h23);
        auto left = [](float x, float y, uint32_t h) {
            return ptx::cvt_bf16x2(x - __uint_as_float(h << 16), y - __uint_as_float(h & 0xffff0000u));
        };
        ptx::st_shared(p_mine + kMaxGroup * SM::kPPitch, left(p0, p1, h01));
        ptx::st_shared(p_mine + kMaxGroup * SM::kPPitch + 16, left(p2, p3, h23));
        float lsum = (p0 + p1) + (p2 + p3);
        lsum += __shfl_xor_sync(0xffffffffu, lsum, 1);
        lsum += __shfl_xor_sync(0xffffffffu, lsum, 2);
        l_run = l_run * alpha + lsum;
        m_run = m_new;
        if (t == 0) ptx::st_shared(rest + SM::kSum + stat_mine, __float_as_uint(l_run));
        __syncthreads();
        // ---- O = alpha O + P V: rows = heads, the blocks' keys 16 at a time, this warp's D / 8 features.
#pragma unroll
        for (int e = 0; e < NT; ++e) {
            acc[e][0] *= alpha;
            acc[e][1] *= alpha;
            acc[e][2] *= alpha;
            acc[e][3] *= alpha;
        }
#pragma unroll 1
        for (int x = 0; x < blocks; ++x) {
            const int s = (i0 + x) % stages;
            wait_bar(bar_vfull(s), (uint32_t)((i0 + x) / stages) & 1, 3);
            __syncwarp();
            const uint32_t sv = smem_base + (uint32_t)s * SM::kStage + SM::kTile;
            uint32_t pf[4][4], vf[4][2 * NT];
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
                ptx::ldmatrix_x4(p_frag + (uint32_t)(64 * x + 16 * ks) * 2u, pf[ks][0], pf[ks][1], pf[ks][2], pf[ks][3]);
            if constexpr (NT == 2) {
                const int ch = 2 * wid + (lane >> 4);
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) {
                    const int key = 16 * ks + (((lane >> 3) & 1) << 3) + (lane & 7);
                    ptx::ldmatrix_x4_trans(sv + (uint32_t)(ch >> 3) * SM::kSub + (uint32_t)key * 128u +
                                               (uint32_t)(((ch & 7) ^ (key & 7)) << 4),
                                           vf[ks][0], vf[ks][1], vf[ks][2], vf[ks][3]);
                }
            } else {
                const int ch = wid;
#pragma unroll
                for (int ks = 0; ks < 4; ks += 2) {
                    const int key = 16 * ks + ((lane >> 3) << 3) + (lane & 7);
                    ptx::ldmatrix_x4_trans(sv + (uint32_t)key * 128u + (uint32_t)((ch ^ (key & 7)) << 4), vf[ks][0], vf[ks][1],
                                           vf[ks + 1][0], vf[ks + 1][1]);
                }
            }
            // V rows of keys that do not exist may hold anything (0 x NaN would poison O): they are cleared in the
            // fragments.  Only the diagonal block has such rows.
            if (r == 0 && i0 + x == 0) {
                const int keys = (len - 1) % kDecBlock + 1;
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) {
                    const int key0 = 16 * ks + 2 * t;
                    const uint32_t keep0 = (key0 < keys ? 0x0000ffffu : 0u) | (key0 + 1 < keys ? 0xffff0000u : 0u);
                    const uint32_t keep1 = (key0 + 8 < keys ? 0x0000ffffu : 0u) | (key0 + 9 < keys ? 0xffff0000u : 0u);
#pragma unroll
                    for (int e = 0; e < NT; ++e) {
                        vf[ks][2 * e] &= keep0;
                        vf[ks][2 * e + 1] &= keep1;
                    }
                }
            }
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
#pragma unroll
                for (int e = 0; e < NT; ++e)
                    mma_bf16(acc[e], pf[ks][0], pf[ks][1], pf[ks][2], pf[ks][3], vf[ks][2 * e], vf[ks][2 * e + 1]);
        }
        // Once every warp has finished with these blocks, their stages may be loaded again; not if a wait gave up: a barrier
        // whose phase is not over must not be armed again, nor a stage loaded that copies are still on their way to.  (The
        // flag is up for good then, and what waits are left give up at their next look at it.)
        if (i0 + stages < mine) {
            __syncthreads();
            if (wid == 0 && !*abort_flag) fetch(i0 + stages, i0 + stages + per);
            __syncwarp();
        }
    }

    // ---- Thread (g, t) of warp w holds head g, features (D / 8) w + 8 e + 2 t + {0, 1}: pushed to CTA g % R.
    ptx::cluster_wait();
    if (g < G) {
        const uint32_t slot = ((uint32_t)g * inv_R) >> 16, owner = (uint32_t)g - slot * (uint32_t)R;
        const uint32_t dst = ptx::map_shared(rest + SM::kRecv, owner) + ((uint32_t)r * (uint32_t)heads_per_owner + slot) * SM::kRecvRow;
        const uint32_t their_bar = ptx::map_shared(bar_recv, owner);
        // (An infinite V: 0 x infinity in the remainder's product must not turn the first part's infinity into NaN.)
        auto both = [](float hi, float lo) { return fabsf(hi) < INFINITY ? hi + lo : hi; };
#pragma unroll
        for (int e = 0; e < NT; ++e)
            ptx::st_async_v2(dst + (uint32_t)(wid * (D / 8) + 8 * e + 2 * t) * 4u, both(acc[e][0], acc[e][2]),
                             both(acc[e][1], acc[e][3]), their_bar);
        if (wid == 0 && t == 0) {
            float l = 0.f;
            if (mine > 0) {
                float lw[kClusterWarps];
                ptx::ld_shared_v4(rest + SM::kSum + stat_row, lw[0], lw[1], lw[2], lw[3]);
                ptx::ld_shared_v4(rest + SM::kSum + stat_row + 16, lw[4], lw[5], lw[6], lw[7]);
                l = ((lw[0] + lw[1]) + (lw[2] + lw[3])) + ((lw[4] + lw[5]) + (lw[6] + lw[7]));
            }
            ptx::st_async_v2(dst + D * 4u, m_run, l, their_bar);
        }
    }

    // ---- Heads r, r + R, ...: D threads a head, a thread one feature.
    if (heads_here > 0 &&
        !ptx::mbar_wait_bounded_cluster(bar_recv, 0, abort_flag, a.status, 4, a.wait_cycles, (int)PA_ERR_TIMEOUT)) {
        // This CTA's shared memory has to last until every peer's part is in it.  A peer is there after at most two waits for
        // each of its at most 16 blocks, so this is over before its own limit is.  (A second barrier of the cluster would do,
        // but its mere presence cost 0.1 us a call.)
        const long long t0 = clock64(), most = 40 * (a.wait_cycles + 2000000ll);
        while (!ptx::mbar_try_wait_cluster(bar_recv, 0) && clock64() - t0 < most) {
        }
    } else if (heads_here > 0) {
        const int d = tid % D;
        for (int slot = tid / D; slot < heads_here; slot += kClusterThreads / D) {
            const int h = r + slot * R;
            float mr[kRowMaxCluster], lr[kRowMaxCluster], orr[kRowMaxCluster];
#pragma unroll
            for (int x = 0; x < kRowMaxCluster; ++x) {
                const uint32_t src = rest + SM::kRecv + (uint32_t)((x < R ? x : 0) * heads_per_owner + slot) * SM::kRecvRow;
                ptx::ld_shared_v2(src + D * 4u, mr[x], lr[x]);
                orr[x] = __uint_as_float(ptx::ld_shared(src + (uint32_t)d * 4u));
            }
            float m = -INFINITY;
#pragma unroll
            for (int x = 0; x < kRowMaxCluster; ++x)
                if (x < R) m = fmaxf(m, mr[x]);
            float l = 0.f, o = 0.f;
#pragma unroll
            for (int x = 0; x < kRowMaxCluster; ++x) {
                const float wgt = (x < R && mr[x] != -INFINITY) ? ptx::ex2(mr[x] - m) : 0.f;
                l = fmaf(lr[x], wgt, l);
                o = fmaf(orr[x], wgt, o);
            }
            const bool any = m != -INFINITY;  // false: a cache length outside [1, max_len]
            const float out = any ? o / l : 0.f;
            const int64_t oi = ((int64_t)rowid * G + h) * D + d;
            if (a.o_is_f32)
                reinterpret_cast<float *>(a.o)[oi] = out;
            else
                reinterpret_cast<__nv_bfloat16 *>(a.o)[oi] = __float2bfloat16_rn(out);
            if (d == 0) a.lse[(int64_t)rowid * G + h] = any ? (m + log2f(l)) * 0.6931471805599453f : -INFINITY;
        }
    }
    if (*abort_flag && tid == 0) {
        // A wait gave up: leave copies that may still be in flight a bounded time to land before the CTA's shared memory is
        // handed to another CTA.  (Thread 0 waits for every V block itself and meets the other warps behind every K block,
        // so it has seen the flag unless all copies have landed.)
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000ll) {
        }
    }
}

__global__ void decode_block_list_kernel(int64_t len, int32_t W, int32_t S, int32_t *out,
                                         int32_t *count, int32_t capacity)
{
    const LayoutRow row = layout_row((len - 1) / kDecBlock, W, S);
    for (int32_t pos = 0; pos < row.n && pos < capacity; ++pos) out[pos] = (int32_t)layout_entry(row, pos);
    *count = (int32_t)row.n;
}

// One warp: the enumeration of the cluster and row kernels, compacted in lane order.
__global__ void decode_row_block_set_kernel(int64_t len, int32_t W, int32_t S, int32_t *out, int32_t *count,
                                            int32_t capacity)
{
    const int lane = threadIdx.x;
    const int32_t row = (int32_t)((len - 1) / kDecBlock);
    const int32_t cand = row_block_candidate(row, W, S, lane);
    const uint32_t have = __ballot_sync(0xffffffffu, cand >= 0);
    const int pos = __popc(have & ((1u << lane) - 1u));
    if (cand >= 0 && pos < capacity) out[pos] = cand;
    if (lane == 0) *count = __popc(have);
}

// pa_kv_append: a CTA per sequence.  The new token's K and V rows go into the page that holds position
// cache_lens[b], 16 bytes per thread and turn; once every thread has read the old length it grows by one.  A
// sequence whose block table has no valid page for that position is left alone.  (One launch: copying and
// advancing the lengths in two kernels, each waiting for the one before it, cost a decoding step a third launch.)
// kThreads: 128 or, beyond 256 pieces, 1024, since a thread's turns follow one another (64 heads of 128 features, 8
// sequences: 4.6 us with 128 threads, 2.8 with 1024; 8 heads 1.9 and 1.8; one head of 64 features 1.7 and 1.7).
template <int kThreads>
__global__ void __launch_bounds__(kThreads)
kv_append_kernel(const __nv_bfloat16 *k_new, const __nv_bfloat16 *v_new, __nv_bfloat16 *k_pool, __nv_bfloat16 *v_pool,
                 const int32_t *table, int32_t *lens, int32_t table_stride, int32_t n_pages, int32_t Hkv, int32_t D,
                 int64_t k_sp, int64_t k_ss, int64_t k_sh, int64_t v_sp, int64_t v_ss, int64_t v_sh)
{
    pdl_launch_next();
    pdl_wait();
    const int b = blockIdx.x;
    const int per_row = D / 8, pieces = Hkv * per_row;  // 16-byte pieces of K, then of V
    auto piece_of = [&](int x) {
        const bool is_v = x >= pieces;
        return ld16((is_v ? v_new : k_new) + ((int64_t)b * pieces + (is_v ? x - pieces : x)) * 8);
    };
    // A thread's first piece is on its way while the length and then the page are looked up.
    const int first = threadIdx.x;
    uint4 piece = make_uint4(0, 0, 0, 0);
    const int32_t pos = lens[b];
    if (first < 2 * pieces) piece = piece_of(first);
    const int32_t blk = pos / kDecBlock;
    if (pos < 0 || blk >= table_stride) return;
    const int32_t page = table[(int64_t)b * table_stride + blk];
    if (page < 0 || page >= n_pages) return;
    const int slot = pos % kDecBlock;
    for (int x = first; x < 2 * pieces; x += kThreads) {
        const bool is_v = x >= pieces;
        const int y = is_v ? x - pieces : x, hk = y / per_row, c = y % per_row;
        if (x != first) piece = piece_of(x);
        __nv_bfloat16 *dst = is_v ? v_pool + page * v_sp + slot * v_ss + hk * v_sh
                                  : k_pool + page * k_sp + slot * k_ss + hk * k_sh;
        *reinterpret_cast<uint4 *>(dst + 8 * c) = piece;
    }
    __syncthreads();
    if (threadIdx.x == 0) lens[b] = pos + 1;
}

// Window distances + power-of-two distances beyond the window + sink blocks that a row below
// n_rows can have, before any of them coincide or fall off the sequence start: the number of
// candidate slots the cluster and row kernels enumerate (one per lane, so it needs this to be <= 32).
static int64_t row_candidate_slots(int64_t n_rows, int32_t W, int32_t S)
{
    const int64_t w = W > 1 ? W : 1;
    int powers = 0;
    for (int64_t pw = 1; pw <= n_rows - 1; pw *= 2)
        if (pw >= w) ++powers;
    return w + S + powers;
}

// Upper bound on the number of listed blocks of any row below n_rows.
static int max_row_blocks(int64_t n_rows, int32_t W, int32_t S)
{
    // window distances 0 .. w-1, every power of two 2^k >= w with 2^k <= n_rows - 1, sink blocks
    const int64_t bound = row_candidate_slots(n_rows, W, S);
    return (int)(bound < n_rows ? bound : n_rows);
}

// What the checks below need to know about a decode problem, whichever cache form it uses.
struct DecodeShape {
    int32_t batch, n_q_heads, n_kv_heads, head_dim, block, window_blocks, sink_blocks;
    int64_t max_len;
    pa_strides k, v;
    pa_dtype o_dtype;
    float softmax_scale;
};

static pa_status check_decode_shape(const DecodeShape &p)
{
    if (p.batch < 1 || p.n_q_heads < 1 || p.n_kv_heads < 1 || p.max_len < 1)
        return fail(PA_ERR_INVALID_ARG, "batch, head counts and max_len must be positive");
    if (p.window_blocks < 0 || p.sink_blocks < 0)
        return fail(PA_ERR_INVALID_ARG, "window_blocks and sink_blocks must be >= 0");
    if (p.o_dtype != PA_BF16 && p.o_dtype != PA_F32) return fail(PA_ERR_INVALID_ARG, "bad o_dtype");
    if (!(p.softmax_scale >= 0.f) || isinf(p.softmax_scale))
        return fail(PA_ERR_INVALID_ARG, "softmax_scale must be finite and >= 0 (0 = default)");
    if (p.head_dim != 64 && p.head_dim != 128) return fail(PA_ERR_SHAPE, "head_dim must be 64 or 128");
    if (p.block != kDecBlock) return fail(PA_ERR_SHAPE, "block must be 64");
    if (p.n_q_heads % p.n_kv_heads) return fail(PA_ERR_SHAPE, "n_q_heads must be a multiple of n_kv_heads");
    if (p.n_q_heads / p.n_kv_heads > kMaxGroup)
        return fail(PA_ERR_SHAPE, "at most %d query heads per KV head", kMaxGroup);
    if (p.max_len > ((int64_t)1 << 30)) return fail(PA_ERR_SHAPE, "max_len too large (limit 2^30 tokens)");
    if (p.batch > 65535 || p.n_kv_heads > 65535 || p.n_q_heads > 65535)
        return fail(PA_ERR_SHAPE, "batch and head counts must be <= 65535");
    if (p.window_blocks > 4096 || p.sink_blocks > 4096)
        return fail(PA_ERR_SHAPE, "window_blocks and sink_blocks must be <= 4096");
    const pa_strides *st[2] = {&p.k, &p.v};
    for (auto s : st) {
        if (s->seq < p.head_dim || s->head < p.head_dim || s->batch < 0)
            return fail(PA_ERR_SHAPE, "cache strides must be >= head_dim");
        if ((s->seq % 8) || (s->head % 8) || (s->batch % 8))
            return fail(PA_ERR_ALIGNMENT, "cache strides must be multiples of 8 elements (16 bytes)");
        if (s->seq >= ((int64_t)1 << 38) || s->head >= ((int64_t)1 << 38) || s->batch >= ((int64_t)1 << 38))
            return fail(PA_ERR_SHAPE, "cache strides too large for a tensor map");
    }
    return PA_OK;
}

static pa_status shape_of(const pa_decode_params *p, DecodeShape *s)
{
    if (!p) return fail(PA_ERR_INVALID_ARG, "params must be non-null");
    *s = DecodeShape{p->batch, p->n_q_heads, p->n_kv_heads, p->head_dim, p->block, p->window_blocks, p->sink_blocks,
                     p->max_len, p->k, p->v, p->o_dtype, p->softmax_scale};
    return check_decode_shape(*s);
}

static pa_status shape_of(const pa_paged_params *p, DecodeShape *s)
{
    if (!p) return fail(PA_ERR_INVALID_ARG, "params must be non-null");
    if (p->n_pages < 1 || p->max_blocks_per_seq < 1)
        return fail(PA_ERR_INVALID_ARG, "n_pages and max_blocks_per_seq must be positive");
    *s = DecodeShape{p->batch, p->n_q_heads, p->n_kv_heads, p->head_dim, p->block, p->window_blocks, p->sink_blocks,
                     (int64_t)p->max_blocks_per_seq * kDecBlock, p->k, p->v, p->o_dtype, p->softmax_scale};
    if (pa_status st = check_decode_shape(*s)) return st;
    if (p->k.batch < (int64_t)kDecBlock * p->head_dim || p->v.batch < (int64_t)kDecBlock * p->head_dim)
        return fail(PA_ERR_SHAPE, "the page stride must cover a page of %d tokens", kDecBlock);
    return PA_OK;
}

static bool takes_split_k(const DecodeShape &s)
{
    const int64_t rows = (s.max_len + kDecBlock - 1) / kDecBlock;
    return env_switches().decode_path == 1 || row_candidate_slots(rows, s.window_blocks, s.sink_blocks) > 32;
}

static size_t decode_workspace_bytes(const DecodeShape &s)
{
    const int64_t rows = (s.max_len + kDecBlock - 1) / kDecBlock;
    const int chunks = max_row_blocks(rows, s.window_blocks, s.sink_blocks);
    return kDecStatusBytes + (size_t)s.batch * s.n_q_heads * chunks * (s.head_dim + 2) * sizeof(float);
}

static size_t row_smem_bytes(int head_dim, int stages, bool cluster)
{
    if (cluster) return head_dim == 128 ? ClusterSmem<128>::bytes(stages) : ClusterSmem<64>::bytes(stages);
    return head_dim == 128 ? RowSmem<128>::bytes(stages) : RowSmem<64>::bytes(stages);
}

// (The last attribute is the one that lets the kernel start early.)
static cudaLaunchConfig_t row_launch_config(unsigned grid, unsigned threads, int R, size_t smem, cudaLaunchAttribute (&attr)[2])
{
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)R;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1] = pdl_attribute();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cfg;
}

// How many clusters of R CTAs of the cluster kernel the device holds at once.  Asked once per device and kind of launch.
static pa_status resident_clusters(int device, int head_dim, int stages, int R, int *out)
{
    static std::mutex mu;
    static int known[kMaxDevices][2][kRowMaxStages + 1][kRowMaxCluster + 1];  // the number plus one; 0: not asked yet
    std::lock_guard<std::mutex> lock(mu);
    int &n = known[device][head_dim == 128][stages][R];
    if (n == 0) {
        cudaLaunchAttribute attr[2];
        const cudaLaunchConfig_t cfg = row_launch_config((unsigned)R, kClusterThreads, R, row_smem_bytes(head_dim, stages, true), attr);
        int found = 0;
        if (head_dim == 128)
            PA_CUDA_OK(cudaOccupancyMaxActiveClusters(&found, decode_cluster_kernel<128>, &cfg));
        else
            PA_CUDA_OK(cudaOccupancyMaxActiveClusters(&found, decode_cluster_kernel<64>, &cfg));
        n = found + 1;
    }
    *out = n - 1;
    return PA_OK;
}

// The launch shared by every decode entry point.  table == null: contiguous cache.
static pa_status launch_decode(const DecodeShape &p, const void *q, const void *k_cache, const void *v_cache,
                               const int32_t *table, int32_t table_stride, int32_t n_pages,
                               const int32_t *cache_lens, void *o, float *lse, void *workspace,
                               size_t workspace_bytes, void *stream)
{
    if (!q || !k_cache || !v_cache || !cache_lens || !o || !lse)
        return fail(PA_ERR_INVALID_ARG, "q, the caches, cache_lens, o and lse must be non-null");
    if (!aligned16(q) || !aligned16(k_cache) || !aligned16(v_cache) || !aligned16(o))
        return fail(PA_ERR_ALIGNMENT, "q, the caches and o must be 16-byte aligned");
    // (What this launch really touches: the status block, plus the partials on the split-K path.
    // The public entry points hold their callers to the documented size before they get here.)
    const size_t need = takes_split_k(p) ? decode_workspace_bytes(p) : kDecStatusBytes;
    if (!workspace || workspace_bytes < need)
        return fail(PA_ERR_WORKSPACE, "workspace of %zu bytes needed, %zu given", need, workspace_bytes);
    if (!aligned16(workspace)) return fail(PA_ERR_ALIGNMENT, "workspace must be 16-byte aligned");
    DeviceInfo dev;
    if (pa_status s = current_sm100_device(&dev)) return s;

    DecodeArgs a;
    a.q = static_cast<const __nv_bfloat16 *>(q);
    a.k = static_cast<const __nv_bfloat16 *>(k_cache);
    a.v = static_cast<const __nv_bfloat16 *>(v_cache);
    a.lens = cache_lens;
    a.table = table;
    a.table_stride = table_stride;
    a.n_pages = n_pages;
    a.status = static_cast<int32_t *>(workspace);
    a.partial = reinterpret_cast<float *>(static_cast<uint8_t *>(workspace) + kDecStatusBytes);
    a.o = o;
    a.lse = lse;
    a.k_sb = p.k.batch; a.k_ss = p.k.seq; a.k_sh = p.k.head;
    a.v_sb = p.v.batch; a.v_ss = p.v.seq; a.v_sh = p.v.head;
    a.max_len = p.max_len;
    a.batch = p.batch; a.Hq = p.n_q_heads; a.Hkv = p.n_kv_heads;
    a.G = p.n_q_heads / p.n_kv_heads;
    a.W = p.window_blocks; a.S = p.sink_blocks;
    const int64_t rows = (p.max_len + kDecBlock - 1) / kDecBlock;
    a.chunks = max_row_blocks(rows, p.window_blocks, p.sink_blocks);
    a.o_is_f32 = p.o_dtype == PA_F32;
    a.stages = 0;
    const float scale = p.softmax_scale != 0.f ? p.softmax_scale : 1.0f / sqrtf((float)p.head_dim);
    a.scale_log2 = scale * 1.4426950408889634f;
    // Block 0 clears the error code as it starts, a second before any wait can run out; under a caller's limit, which
    // may be shorter than the time from one CTA's start to another's, it is cleared ahead of the kernel.
    const long long wait_cycles = wait_limit_cycles();
    a.wait_cycles = wait_cycles > 0 ? wait_cycles : kRowWaitCycles;
    a.clear_status = wait_cycles <= 0;

    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (!a.clear_status) PA_CUDA_OK(cudaMemsetAsync(a.status, 0, sizeof(int32_t), st));
    const EnvSwitches env = env_switches();
    a.fixed_chunks = 0;
    a.R = 1;
    a.items = 0;
    // Rows whose block set fits one warp's lanes take the cluster or the row kernel.
    if (!takes_split_k(p)) {
        const int64_t rows_in_call = (int64_t)a.batch * a.Hkv;
        const int max_R = a.chunks < kRowMaxCluster ? a.chunks : kRowMaxCluster;
        const int64_t persistent_ctas = (env.decode_ctas_per_sm ? env.decode_ctas_per_sm : 2) * (int64_t)dev.sms;
        // Stages: 64 KB of blocks in flight per CTA, and no more than a CTA has blocks.
        // (two stages measured 1-3 % faster than three at batch 64 and 256, head_dim 128)
        auto stages_of = [&](int64_t ctas, bool cluster_form) {
            const int64_t blocks_per_cta = ((int64_t)a.chunks * rows_in_call + ctas - 1) / ctas;
            int n = env.decode_stages != 0 ? env.decode_stages : p.head_dim == 128 ? 2 : 4;
            if (n > kRowMaxStages) n = kRowMaxStages;
            if (n > blocks_per_cta) n = (int)blocks_per_cta;
            if (n < 1) n = 1;
            while (n > 1 && row_smem_bytes(p.head_dim, n, cluster_form) > (size_t)kRowMaxSmem) --n;
            return n;
        };
        if (pa_status s = device_once(dev.device, ONCE_DECODE_ATTR, [] {
                constexpr cudaFuncAttribute kSmem = cudaFuncAttributeMaxDynamicSharedMemorySize;
                cudaError_t e = cudaSuccess;
                for (auto *kernel : {decode_row_kernel<128, true>, decode_row_kernel<128, false>, decode_row_kernel<64, true>,
                                     decode_row_kernel<64, false>, decode_cluster_kernel<128>, decode_cluster_kernel<64>})
                    e = first_error(e, cudaFuncSetAttribute(kernel, kSmem, kRowMaxSmem));
                return e;
            }))
            return s;
        // Small calls (latency-bound): a cluster of R CTAs per row, all resident at once.  Larger calls
        // (bandwidth-bound): a persistent grid of two CTAs per SM over the rows.  The line lies where a row
        // still gets two of the resident CTAs: 4000 tokens, G = 7, head_dim 128 take 6.8 us at 80 rows in clusters
        // of three, 9.1 at 148 in clusters of two, 13.8 (clusters of one) and 11.3 (persistent form) at 160.
        bool cluster = rows_in_call * 2 <= persistent_ctas;
        if (env.decode_path == 2) cluster = true;
        if (env.decode_path == 3) cluster = false;
        int R = env.decode_cluster, fit = 0;  // fit: clusters of R CTAs that the device holds at once
        if (cluster && R == 0) {
            // As many CTAs per row as run all at once: a second wave of clusters nearly doubles the call's latency
            // (with an earlier kernel, 4000 tokens, G = 7, head_dim 128: 74 rows in clusters of four 13.0 us, of three
            // 8.2).  How many clusters fit is asked of the device: all CTAs of a cluster lie within one GPU processing
            // cluster, which may leave places that no further cluster fits in.
            R = (int)(persistent_ctas / rows_in_call);
            if (R > max_R) R = max_R;
            for (; R > 1; --R) {
                const int stages = stages_of(rows_in_call * R, true);
                if (pa_status s = resident_clusters(dev.device, p.head_dim, stages, R, &fit)) return s;
                if (rows_in_call <= fit) break;
            }
        }
        // (Large calls: one chunk per row.  Finer items balance the SMs better on paper but pay more per item
        // than they gain, and need the merge kernel.)
        if (R < 1) R = 1;
        if (R > max_R) R = max_R;
        // A row in one piece has nothing to merge with, and nothing that eight warps could share (one block, G = 7,
        // head_dim 128: 4.3 to 5.9 us in the cluster form, 3.4 to 4.6 without).
        if (R == 1 && env.decode_path != 2) cluster = false;
        const bool parts = !cluster && R > 1;
        a.R = R;
        a.items = rows_in_call * R;
        const int64_t grid = cluster ? a.items : (a.items < persistent_ctas ? a.items : persistent_ctas);
        if (a.items > 0x3fffffff) return fail(PA_ERR_SHAPE, "too many work items (%lld)", (long long)a.items);
        a.stages = stages_of(grid, cluster);
        // Started early, clusters take places as the CTAs of the kernel before leave them, one by one, and what is left
        // in between may be of no use to a cluster until more have ended.  A call that needs nearly all places starts
        // on the empty device instead, about 1 us later.  Where that begins to pay was measured for each size, early
        // and late in us (148 SMs: 93 clusters of three fit, 71 of four, 56 of five).  Clusters of three, 128 features, G = 7,
        // 4000 tokens: 7.4 and 8.0 at 87 rows, 8.2 and 8.0 at 88, 9.4 and 8.0 at 90 (G = 8, 30000 tokens: 7.8 and 8.9 at 90, 9.4 and
        // 8.9 at 93); 64 features, G = 4: 5.4 and 6.4 at 90, 6.1 and 6.4 at 92, 6.7 and 6.4 at 93.  Of four and five 6.8 and 7.7 at
        // 70, 8.1 and 7.7 at 71, 5.8 and 6.3 at 55, 6.3 and 6.3 at 56 (64 features 5.6 and 6.3 at 71, 5.7 and 5.2 at 56).  Of six to
        // eight never clearly: 5.4 and 6.2 at 45, 6.2 and 5.9 at 37, 6.1 and 5.9 at 33.  A row of one head is merged by one of its
        // CTAs, the others leave before it, which spoils more places: of three 7.9 and 7.1 at 85, 8.9 and 7.1 at 88 (64
        // features 6.6 and 6.8, 8.5 and 6.8), of five 5.8 and 5.7 at 50, 6.9 and 5.7 at 51 (7.2 and 6.2, 7.6 and 6.2).  Pairs fit
        // in any order.
        const bool full = a.G == 1 && (R == 3 || R == 5) ? rows_in_call * 100 > (int64_t)fit * 91
                          : R == 3 && p.head_dim == 128  ? rows_in_call * 20 > (int64_t)fit * 19
                                                         : R <= 5 && rows_in_call == fit;
        const bool early = !(cluster && R > 2 && fit > 0 && full);

        // Tensor maps over the cache: (feature, token, head, batch or page), one 64 x 64 box per copy.
        CUtensorMap tmK, tmV;
        const bool paged = table != nullptr;
        TensorMapKey kk = {k_cache, paged ? (int64_t)kDecBlock : p.max_len, p.k.seq, p.k.head, p.k.batch, dev.device,
                           p.head_dim, p.n_kv_heads, paged ? n_pages : p.batch, 1, kDecBlock, 0};
        TensorMapKey kv = {v_cache, paged ? (int64_t)kDecBlock : p.max_len, p.v.seq, p.v.head, p.v.batch, dev.device,
                           p.head_dim, p.n_kv_heads, paged ? n_pages : p.batch, 1, kDecBlock, 0};
        if (pa_status s = get_tensor_map(kk, "k_cache", &tmK)) return s;
        if (pa_status s = get_tensor_map(kv, "v_cache", &tmV)) return s;

        if (parts) {
            a.chunks = R;  // the partials of a row are its R chunks
            a.fixed_chunks = R;
        }
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg =
            row_launch_config((unsigned)grid, cluster ? kClusterThreads : kRowThreads, cluster ? R : 1,
                              row_smem_bytes(p.head_dim, a.stages, cluster), attr);
        cfg.stream = st;
        if (!early) cfg.numAttrs = 1;
        auto kernel_of = [&](auto d) {
            constexpr int D = decltype(d)::value;
            return cluster ? decode_cluster_kernel<D> : parts ? decode_row_kernel<D, true> : decode_row_kernel<D, false>;
        };
        auto *kernel = p.head_dim == 128 ? kernel_of(std::integral_constant<int, 128>()) : kernel_of(std::integral_constant<int, 64>());
        PA_CUDA_OK(cudaLaunchKernelEx(&cfg, kernel, tmK, tmV, a));
        if (!parts) return PA_OK;
    } else {
        const dim3 grid1((unsigned)a.chunks, (unsigned)a.Hkv, (unsigned)a.batch);
        if (p.head_dim == 128)
            decode_block_kernel<128><<<grid1, kDecThreads, 0, st>>>(a);
        else
            decode_block_kernel<64><<<grid1, kDecThreads, 0, st>>>(a);
        PA_CUDA_OK(cudaGetLastError());
    }

    const dim3 heads((unsigned)a.Hq, (unsigned)a.batch, 1);
    if (p.head_dim == 128)
        PA_CUDA_OK(launch_pdl(decode_combine_kernel<128>, heads, 128, 0, st, a));
    else
        PA_CUDA_OK(launch_pdl(decode_combine_kernel<64>, heads, 64, 0, st, a));
    return PA_OK;
}

}  // namespace pa

extern "C" size_t pa_decode_workspace_bytes(const pa_decode_params *p)
{
    using namespace pa;
    DecodeShape s;
    if (shape_of(p, &s) != PA_OK) return 0;
    return decode_workspace_bytes(s);
}

extern "C" pa_status pa_decode(const pa_decode_params *p, const void *q, const void *k_cache,
                               const void *v_cache, const int32_t *cache_lens, void *o,
                               float *lse, void *workspace, size_t workspace_bytes, void *stream)
{
    using namespace pa;
    clear_error();
    DecodeShape s;
    if (pa_status st = shape_of(p, &s)) return st;
    const size_t need = decode_workspace_bytes(s);
    if (!workspace || workspace_bytes < need)
        return fail(PA_ERR_WORKSPACE, "workspace of %zu bytes needed, %zu given", need, workspace_bytes);
    return launch_decode(s, q, k_cache, v_cache, nullptr, 0, 0, cache_lens, o, lse, workspace, workspace_bytes, stream);
}

extern "C" size_t pa_decode_paged_workspace_bytes(const pa_paged_params *p)
{
    using namespace pa;
    DecodeShape s;
    if (shape_of(p, &s) != PA_OK) return 0;
    return decode_workspace_bytes(s);
}

extern "C" pa_status pa_decode_paged(const pa_paged_params *p, const void *q, const void *k_pool,
                                     const void *v_pool, const int32_t *block_table,
                                     const int32_t *cache_lens, void *o, float *lse, void *workspace,
                                     size_t workspace_bytes, void *stream)
{
    using namespace pa;
    clear_error();
    DecodeShape s;
    if (pa_status st = shape_of(p, &s)) return st;
    if (!block_table) return fail(PA_ERR_INVALID_ARG, "block_table must be non-null");
    const size_t need = decode_workspace_bytes(s);
    if (!workspace || workspace_bytes < need)
        return fail(PA_ERR_WORKSPACE, "workspace of %zu bytes needed, %zu given", need, workspace_bytes);
    return launch_decode(s, q, k_pool, v_pool, block_table, p->max_blocks_per_seq, p->n_pages, cache_lens, o, lse,
                         workspace, workspace_bytes, stream);
}

extern "C" pa_status pa_kv_append(const pa_paged_params *p, const void *k_new, const void *v_new, void *k_pool,
                                  void *v_pool, const int32_t *block_table, int32_t *cache_lens, void *stream)
{
    using namespace pa;
    clear_error();
    DecodeShape s;
    if (pa_status st = shape_of(p, &s)) return st;
    if (!k_new || !v_new || !k_pool || !v_pool || !block_table || !cache_lens)
        return fail(PA_ERR_INVALID_ARG, "k_new, v_new, the pools, block_table and cache_lens must be non-null");
    if (!aligned16(k_new) || !aligned16(v_new) || !aligned16(k_pool) || !aligned16(v_pool))
        return fail(PA_ERR_ALIGNMENT, "k_new, v_new and the pools must be 16-byte aligned");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    auto launch = [&](auto kernel, unsigned threads) {
        return launch_pdl(kernel, dim3((unsigned)p->batch), threads, 0, st, static_cast<const __nv_bfloat16 *>(k_new),
                          static_cast<const __nv_bfloat16 *>(v_new), static_cast<__nv_bfloat16 *>(k_pool),
                          static_cast<__nv_bfloat16 *>(v_pool), block_table, cache_lens, p->max_blocks_per_seq, p->n_pages,
                          p->n_kv_heads, p->head_dim, p->k.batch, p->k.seq, p->k.head, p->v.batch, p->v.seq, p->v.head);
    };
    const int pieces = 2 * p->n_kv_heads * (p->head_dim / 8);
    if (pieces <= 256) PA_CUDA_OK(launch(kv_append_kernel<128>, 128));
    else PA_CUDA_OK(launch(kv_append_kernel<1024>, 1024));
    return PA_OK;
}

extern "C" pa_status pa_decode_status(const void *workspace, void *stream, int32_t *detail)
{
    using namespace pa;
    clear_error();
    if (!workspace) return fail(PA_ERR_INVALID_ARG, "workspace must be non-null");
    int32_t host[2] = {0, 0};
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    PA_CUDA_OK(cudaMemcpyAsync(host, workspace, sizeof host, cudaMemcpyDeviceToHost, st));
    PA_CUDA_OK(cudaStreamSynchronize(st));
    if (detail) *detail = host[1];
    if (host[0] == (int32_t)PA_ERR_TIMEOUT)
        return fail(PA_ERR_TIMEOUT, "a bounded wait inside the decode kernel ran out (wait id %d)", host[1]);
    if (host[0] != 0) return fail(PA_ERR_CUDA, "unexpected device status %d", host[0]);
    return PA_OK;
}

extern "C" pa_status pa_decode_block_list(int64_t cache_len, int32_t block, int32_t window_blocks,
                                          int32_t sink_blocks, int32_t *out_blocks,
                                          int32_t *out_count, int32_t capacity, void *stream)
{
    using namespace pa;
    clear_error();
    if (cache_len < 1) return fail(PA_ERR_INVALID_ARG, "cache_len must be >= 1");
    if (block != kDecBlock) return fail(PA_ERR_SHAPE, "block must be 64");
    if (window_blocks < 0 || sink_blocks < 0 || capacity < 1 || !out_blocks || !out_count)
        return fail(PA_ERR_INVALID_ARG, "bad window/sink/capacity or null output");
    decode_block_list_kernel<<<1, 1, 0, static_cast<cudaStream_t>(stream)>>>(
        cache_len, window_blocks, sink_blocks, out_blocks, out_count, capacity);
    PA_CUDA_OK(cudaGetLastError());
    return PA_OK;
}

extern "C" pa_status pa_decode_row_block_set(int64_t cache_len, int32_t block, int32_t window_blocks,
                                             int32_t sink_blocks, int32_t *out_blocks, int32_t *out_count,
                                             int32_t capacity, void *stream)
{
    using namespace pa;
    clear_error();
    if (cache_len < 1 || cache_len > ((int64_t)1 << 30)) return fail(PA_ERR_INVALID_ARG, "cache_len must be in [1, 2^30]");
    if (block != kDecBlock) return fail(PA_ERR_SHAPE, "block must be 64");
    if (window_blocks < 0 || sink_blocks < 0 || capacity < 32 || !out_blocks || !out_count)
        return fail(PA_ERR_INVALID_ARG, "bad window/sink, capacity < 32 or null output");
    const int64_t rows = (cache_len + kDecBlock - 1) / kDecBlock;
    if (row_candidate_slots(rows, window_blocks, sink_blocks) > 32)
        return fail(PA_ERR_SHAPE, "window + sink + power-of-two candidates exceed 32: such rows take the split-K path");
    decode_row_block_set_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(
        cache_len, window_blocks, sink_blocks, out_blocks, out_count, capacity);
    PA_CUDA_OK(cudaGetLastError());
    return PA_OK;
}

// ------------------------------------------------------------------------------------------
// pa_decode_static: the same decode, for callers that cannot allocate device memory.
//
// The workspace (status block and split-K partial results) is a fixed array that is part of the
// library image instead of a caller-provided buffer.  The array's name is only a host-side handle
// in host code; the real device address is looked up once per device with cudaGetSymbolAddress
// (with that device current) and then handed to the kernels like any other pointer.
// ------------------------------------------------------------------------------------------
namespace pa {

static __device__ __align__(256) unsigned char g_decode_static_scratch[PA_DECODE_STATIC_SCRATCH_BYTES];

static std::mutex g_static_mu;
static void *g_static_ptr[kMaxDevices] = {};

// Device address of the scratch array on the current device (looked up on first use).
static pa_status static_scratch_address(void **out)
{
    int dev = 0;
    PA_CUDA_OK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices)
        return fail(PA_ERR_UNSUPPORTED, "device index %d is beyond the %d devices supported", dev, kMaxDevices);
    std::lock_guard<std::mutex> lock(g_static_mu);
    if (!g_static_ptr[dev]) {
        void *ptr = nullptr;
        PA_CUDA_OK(cudaGetSymbolAddress(&ptr, g_decode_static_scratch));
        if (!ptr) return fail(PA_ERR_CUDA, "cudaGetSymbolAddress returned a null address");
        g_static_ptr[dev] = ptr;
    }
    *out = g_static_ptr[dev];
    return PA_OK;
}

}  // namespace pa

extern "C" pa_status pa_decode_static(const pa_decode_params *p, const void *q, const void *k_cache,
                                      const void *v_cache, const int32_t *cache_lens, void *o,
                                      float *lse, void *stream)
{
    using namespace pa;
    clear_error();
    DecodeShape s;
    if (pa_status st = shape_of(p, &s)) return st;
    // The single-launch path keeps only its status block in the workspace; the partial results
    // of the two-kernel path are what has to fit the built-in array.
    const size_t need = takes_split_k(s) ? decode_workspace_bytes(s) : kDecStatusBytes;
    if (need > (size_t)PA_DECODE_STATIC_SCRATCH_BYTES)
        return fail(PA_ERR_WORKSPACE,
                    "this problem needs %zu bytes of split-K scratch but the built-in array holds %zu; "
                    "use pa_decode with a caller-allocated workspace", need,
                    (size_t)PA_DECODE_STATIC_SCRATCH_BYTES);
    void *scratch = nullptr;
    if (pa_status st = static_scratch_address(&scratch)) return st;
    return launch_decode(s, q, k_cache, v_cache, nullptr, 0, 0, cache_lens, o, lse, scratch,
                         (size_t)PA_DECODE_STATIC_SCRATCH_BYTES, stream);
}
