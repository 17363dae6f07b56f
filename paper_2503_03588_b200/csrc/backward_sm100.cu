// Backward pass of the block-sparse attention (derivatives of Eq. (1), Section 3.1, under the
// key-block lists of Algorithm 1, Section 3.3) on the sm_100a tensor cores, head_dim 64 and 128.
//
// Two persistent kernels with the same skeleton:
//   warp 0       TMA producer (bf16 tiles, 128-byte swizzle, into rings of shared-memory stages)
//   warp 1       tcgen05 issuer of S (one elected lane)
//   warp 2       tensor-memory allocation, issuer of dP
//   warp 3       issuer of the second products
//   warps 4-19   four compute warpgroups
//   warps 20-23  epilogue: an item's finished accumulators out of tensor memory and out to global memory
// Work items are drawn from a counter in memory, by the producer (dQ) or by warp 20 (dK / dV), and handed to the
// other warps through a small ring in shared memory.
// A step is one (query block, key block) pair for a pair of query heads stacked on the 64 tokens of the query
// block: a 128-row tile, as in the forward kernel.  Per step the tensor cores produce S = Q K^T and dP = dO V^T
// (fp32, tensor memory); the compute warps (thread = tile row = TMEM lane) turn them into P = exp2(S scale
// log2e - LSE log2e) and dS = P (dP - delta), rounded to bf16; the second products accumulate in tensor memory.
//
//   dq_kernel   an item is a (query block, head pair): walks the row's key blocks; dS goes back
//               into tensor memory as the A operand of dQ += dS K (128 x D accumulator)
//   dkv_kernel  an item is a (chunk of a key block's listing query blocks, KV head): walks the chunk for every
//               head pair of the group; P and dS go to shared memory as the B operands of dV^T += dO^T P and
//               dK^T += Q^T dS (feature x key accumulators: the A operands are the dO and Q tiles read
//               feature-major)
//
// The dK / dV kernel is launched first, the dQ kernel fills the places that its last items leave.
// Every barrier wait is bounded; a wait that runs out records PA_ERR_TIMEOUT in the status block,
// raises a CTA-wide abort flag, every role leaves its loop and the CTA ends after a bounded pause.
#include <cuda.h>
#include <cuda_bf16.h>
#include <math.h>

#include "backward.cuh"
#include "sm100_ptx.cuh"
#include "tensor_map.cuh"

// Registers per thread by role (control, compute, epilogue warps).  A warpgroup asking for more than the pool
// holds would wait for ever: both kernels start 768 threads x 80.  (48 / 96 / 48 for both spills more, dK / dV
// not at all now.  Backward pass, two runs each: 4001 tokens, 28 / 4 heads, 154.0 and 154.6 us against 151.8 and
// 151.9; 4 x 4096 tokens, 8 / 8 heads, 342 and 344 against 332 and 333; 2 x 8K tokens, 16 / 4 heads of 64 features,
// 270 and 265 against 260 and 254.)
#define PA_DQ_REG_CTRL 40
#define PA_DQ_REG_COMP 96
#define PA_DQ_REG_EPI 56
static_assert(4 * PA_DQ_REG_CTRL + 16 * PA_DQ_REG_COMP + 4 * PA_DQ_REG_EPI <= 24 * 80,
              "register split exceeds the CTA's registers");
#define PA_DKV_REG_CTRL 64
#define PA_DKV_REG_COMP 88
#define PA_DKV_REG_EPI 64
static_assert(4 * PA_DKV_REG_CTRL + 16 * PA_DKV_REG_COMP + 4 * PA_DKV_REG_EPI <= 24 * 80,
              "register split exceeds the CTA's registers");

namespace pa {

constexpr int kTcThreads = 768;
constexpr int kCompWarps = 16;
constexpr uint32_t kTcTmemCols = 512;
constexpr long long kBwdWaitCycles = 4000000000ll;
constexpr uint32_t kRowTile = 128 * 128;   // 128 rows x 64 features: one 128-byte-wide half of a Q or dO tile
constexpr uint32_t kKeyTile = 64 * 128;    // 64 keys x 64 features: one half of a K or V block
// High word of every shared-memory descriptor: 1024 bytes between 8-row groups, version 1, 128-byte swizzle.
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
constexpr uint32_t kItemRing = 4;          // items the producer may be ahead
constexpr uint32_t kBarBytes = 512;        // barriers; the struct below follows
constexpr uint32_t kBarArea = 1024;

// Instruction descriptor (kind::f16, bf16 operands, fp32 accumulation) with both major bits.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, int a_mn, int b_mn)
{
    return ptx::idesc_bf16_f32(M, N, b_mn) | ((uint32_t)a_mn << 15);
}

// A work item as the producer publishes it.  blk: the query block (dQ) or key block (dK / dV); n: how many blocks
// its row or chunk lists, from e0 on (negative: there are no more items); parts: chunks of the key block;
// first: the first block listed (dK / dV).
struct __align__(16) BwdItem {
    int32_t blk, n, e0, hk, b, hp, parts, first;
};
struct BwdTail {
    BwdItem items[kItemRing];
    uint32_t tmem;
    int abort_flag;
};
static_assert(kBarBytes + sizeof(BwdTail) <= kBarArea, "barrier area");

// P = exp2(S scale - lse2) of a pair of keys.
__device__ __forceinline__ uint64_t bwd_p2(uint32_t s0, uint32_t s1, uint64_t scale2, uint64_t neg_lse2)
{
    float y0, y1;
    ptx::unpack_f32x2(ptx::fma_f32x2(ptx::pack_f32x2(__uint_as_float(s0), __uint_as_float(s1)), scale2, neg_lse2), y0, y1);
    return ptx::pack_f32x2(ptx::ex2(y0), ptx::ex2(y1));
}
// P of 32 keys, as packed pairs; keys beyond `lim` (causal term of the diagonal pair) are 0.
__device__ __forceinline__ void bwd_p(uint32_t (&s)[32], bool diag, int lim, uint64_t scale2, uint64_t neg_lse2,
                                      uint64_t (&p)[16])
{
    if (diag) {
#pragma unroll
        for (int x = 0; x < 32; ++x)
            if (x > lim) s[x] = 0xff800000u;
    }
#pragma unroll
    for (int x = 0; x < 16; ++x) p[x] = bwd_p2(s[2 * x], s[2 * x + 1], scale2, neg_lse2);
}
__device__ __forceinline__ uint32_t bwd_cvt(uint64_t v)
{
    float x, y;
    ptx::unpack_f32x2(v, x, y);
    return ptx::cvt_bf16x2(x, y);
}
// dS = P (dP - delta) of a pair of keys.
__device__ __forceinline__ uint64_t bwd_ds(uint64_t p, uint32_t dp0, uint32_t dp1, uint64_t neg_delta2)
{
    return ptx::mul_f32x2(p, ptx::add_f32x2(ptx::pack_f32x2(__uint_as_float(dp0), __uint_as_float(dp1)), neg_delta2));
}
// Lane t of every four lanes holds M[t][0..3] and gets M[0..3][t].
__device__ __forceinline__ void transpose_quad(uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3, int lane)
{
    auto exchange = [&](uint32_t &lo, uint32_t &hi, int d) {
        const bool upper = lane & d;
        const uint32_t got = __shfl_xor_sync(0xffffffffu, upper ? lo : hi, d);
        (upper ? lo : hi) = got;
    };
    exchange(r0, r1, 1);
    exchange(r2, r3, 1);
    exchange(r0, r2, 2);
    exchange(r1, r3, 2);
}
// -LSE in base 2; a row without weights (beyond the sequence, padding head, empty row) gets -inf: P = 0.
__device__ __forceinline__ float bwd_neg_lse2(float lse)
{
    return (lse == -INFINITY || lse == INFINITY) ? -INFINITY : -lse * 1.4426950408889634f;
}

// Neither kernel needs what the other writes.  The dK / dV kernel, whose items are larger, goes first, and the dQ kernel's
// CTAs start as places become free, beside its last items: the former lets the latter start once it has itself waited
// for the preparation, and says so in the status block, and the latter is over only when the former is.  (Measured
// against dQ first and one after the other, whole backward pass in a loop, 28 / 4 heads: 2K tokens 101 -> 81 us, 4001
// 164 -> 156, 32K 1620 -> 1560; 600 tokens, 2 heads of 64 features 23.1 -> 16.3.  dQ first and dK / dV beside its last
// items: 96, 159, 1590 and 17.9.)
__device__ __forceinline__ void say_prepared(const BackwardArgs &a)
{
    if (blockIdx.x == 0 && threadIdx.x == 0)
        asm volatile("st.release.gpu.global.s32 [%0], %1;\n" ::"l"(a.status + kBwdPrepared), "r"(1) : "memory");
}
// Reading the word orders what the preparation wrote before anything read behind this.  (Were it not there, waiting for
// the kernel before would do.)
__device__ __forceinline__ void expect_prepared(const BackwardArgs &a)
{
    int32_t prepared;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];\n" : "=r"(prepared) : "l"(a.status + kBwdPrepared) : "memory");
    if (prepared != 1) pdl_wait();
}

// ------------------------------------------------------------------------------------- dQ
// A step's way is long and serial: S, dP, a warpgroup's loads, exponentials and stores, dQ, some 4500 cycles of
// which the tensor cores work 1024.  So four steps are under way at a time, a warpgroup each.  Tensor memory
// decides the rest: S has four buffers (dS goes over the S it was made from), dP two, which a warpgroup
// therefore loads whole (64 registers a thread) before it works through S 16 keys at a time.  K stays in its
// ring until dQ has read it, V only until dP has.  Q and dO have one buffer each with head_dim 128: the next
// item's tiles arrive while the last steps are computed and their dQ products run.  With head_dim 64, whose
// steps are shorter than that, two.  Bound by the issue of S and dP (1300 clk a step) and by the 128 KB that an
// item starts with.  Measured, 28 / 4 heads at 32K tokens: 524 us at full clocks, where all four warpgroups on
// one step of two key blocks took 583; 64 features, 16 / 4 heads, 2 x 8K tokens: 87 us against 106, 82 with the
// second pair of Q and dO buffers.
template <int D>
struct DqCfg {
    static constexpr int kDH = D / 64;
    static constexpr int kKStages = D == 128 ? 6 : 8, kVStages = D == 128 ? 3 : 4, kRowBufs = D == 128 ? 1 : 2;
    static constexpr uint32_t kTile = kDH * kRowTile, kBlkTile = kDH * kKeyTile;
    static constexpr uint32_t kQ = 0, kG = kTile;  // (further buffers 2 kTile apart)
    static constexpr uint32_t kK = kRowBufs * 2 * kTile, kV = kK + kKStages * kBlkTile;
    static constexpr uint32_t kOut = kV + kVStages * kBlkTile;  // per epilogue warp a patch of 32 rows x 32 fp32
    static constexpr uint32_t kBars = kOut + 4 * 4096;
    static constexpr uint32_t kAlloc = kBars + kBarArea + 1024;
    static_assert(kAlloc <= 227 * 1024, "shared memory budget");
    enum : uint32_t {
        Q_FULL, Q_EMPTY = Q_FULL + kRowBufs, G_FULL = Q_EMPTY + kRowBufs, G_EMPTY = G_FULL + kRowBufs,
        K_FULL = G_EMPTY + kRowBufs, K_EMPTY = K_FULL + kKStages,
        V_FULL = K_EMPTY + kKStages, V_EMPTY = V_FULL + kVStages,
        S_FULL = V_EMPTY + kVStages, DP_FULL = S_FULL + 4,   // [warpgroup]
        DP_TAKEN = DP_FULL + 4,                              // [step parity]: dP is in registers
        DS_FULL = DP_TAKEN + 2, DS_FREE = DS_FULL + 4,       // [warpgroup]: dS is in tensor memory / dQ += dS K has read it
        DQ_DONE = DS_FREE + 4,               // the item's last dQ += dS K has completed
        DQ_FREE,                             // the epilogue warps have read dQ out of tensor memory
        ITEM_FULL, ITEM_EMPTY = ITEM_FULL + kItemRing, COUNT = ITEM_EMPTY + kItemRing
    };
    static_assert(COUNT * 8 <= kBarBytes, "barrier area");
    // Tensor memory columns: S at 64 g (dS, bf16 pairs, over its first half), dP at 256 + 64 (step parity), dQ.
    static constexpr uint32_t kColDp = 256, kColDq = 384;
};

template <int D>
__global__ void __launch_bounds__(kTcThreads, 1)
dq_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmG,
          const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
          const __grid_constant__ CUtensorMap tmDq, const BackwardArgs a, const uint32_t n_items)
{
    using C = DqCfg<D>;
    constexpr int DH = C::kDH;
    constexpr uint32_t NK = C::kKStages, NV = C::kVStages, NR = C::kRowBufs;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (smem_base - ptx::smem_u32(smem_raw));
    const uint32_t bars = smem_base + C::kBars;
    BwdTail *tail = reinterpret_cast<BwdTail *>(smem + C::kBars + kBarBytes);
    volatile int *abort_flag = &tail->abort_flag;
    auto bar = [&](uint32_t idx) { return bars + idx * 8u; };
    auto wait_bar = [&](uint32_t b_, uint32_t parity, int code) {
        return ptx::mbar_wait_bounded(b_, parity, abort_flag, a.status, code, a.wait_cycles, (int)PA_ERR_TIMEOUT);
    };
    auto wait_warp = [&](uint32_t b_, uint32_t parity, int code) {
        return __all_sync(0xffffffffu, wait_bar(b_, parity, code)) != 0;
    };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // Item number k of this CTA, read by every warp but the producer's.
    auto read_item = [&](uint32_t k, BwdItem &w) {
        if (!wait_warp(bar(C::ITEM_FULL + k % kItemRing), (k / kItemRing) & 1, 1)) return false;
        w = tail->items[k % kItemRing];
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(bar(C::ITEM_EMPTY + k % kItemRing));
        return true;
    };

    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < NR; ++s) {
            ptx::mbar_init(bar(C::Q_FULL + s), 1);
            ptx::mbar_init(bar(C::Q_EMPTY + s), 1);
            ptx::mbar_init(bar(C::G_FULL + s), 1);
            ptx::mbar_init(bar(C::G_EMPTY + s), 1);
        }
        for (uint32_t s = 0; s < NK; ++s) {
            ptx::mbar_init(bar(C::K_FULL + s), 1);
            ptx::mbar_init(bar(C::K_EMPTY + s), 1);
        }
        for (uint32_t s = 0; s < NV; ++s) {
            ptx::mbar_init(bar(C::V_FULL + s), 1);
            ptx::mbar_init(bar(C::V_EMPTY + s), 1);
        }
        for (int g = 0; g < 4; ++g) {
            ptx::mbar_init(bar(C::S_FULL + g), 1);
            ptx::mbar_init(bar(C::DP_FULL + g), 1);
            ptx::mbar_init(bar(C::DS_FULL + g), 4);
            ptx::mbar_init(bar(C::DS_FREE + g), 1);
        }
        ptx::mbar_init(bar(C::DP_TAKEN), 4);
        ptx::mbar_init(bar(C::DP_TAKEN + 1), 4);
        ptx::mbar_init(bar(C::DQ_DONE), 1);
        ptx::mbar_init(bar(C::DQ_FREE), 4);
        for (uint32_t r = 0; r < kItemRing; ++r) {
            ptx::mbar_init(bar(C::ITEM_FULL + r), 1);
            ptx::mbar_init(bar(C::ITEM_EMPTY + r), kTcThreads / 32 - 1);
        }
        tail->abort_flag = 0;
        ptx::fence_barrier_init();
        ptx::fence_proxy_async_smem();
    }
    if (warp == 2) {
        ptx::tmem_alloc(ptx::smem_u32(&tail->tmem), kTcTmemCols);
        ptx::tmem_relinquish();
    }
    if (a.early) pdl_launch_next();
    expect_prepared(a);  // (this kernel runs beside the dK / dV kernel)
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = tail->tmem;

    if (warp < 4) ptx::setmaxnreg_dec<PA_DQ_REG_CTRL>();
    if (warp == 0) {
        // -------------------------------------------------------------- TMA producer
        if (lane == 0) {
            ptx::prefetch_tensormap(&tmQ);
            ptx::prefetch_tensormap(&tmG);
            ptx::prefetch_tensormap(&tmK);
            ptx::prefetch_tensormap(&tmV);
            // Items: query blocks from the last (longest row) to the first, and within a query block the head
            // pairs and batch entries; each CTA starts with its own number and draws further ones.
            uint32_t it = blockIdx.x;
            auto next_item = [&](BwdItem &w) {
                w.n = -1;
                if (it >= n_items) return;
                const uint32_t per_row = (uint32_t)(a.Hkv * a.npairs * a.batch);
                const uint32_t x = it / per_row, yz = it - x * per_row;
                const uint32_t bb = yz / (uint32_t)(a.Hkv * a.npairs), hkp = yz - bb * (uint32_t)(a.Hkv * a.npairs);
                w.blk = a.nqb - 1 - (int32_t)x;
                w.b = (int32_t)bb;
                w.hk = (int32_t)(hkp / (uint32_t)a.npairs);
                w.hp = (int32_t)(hkp % (uint32_t)a.npairs);
                w.e0 = a.row_ptr[w.blk];
                w.n = a.row_ptr[w.blk + 1] - w.e0;
                it = gridDim.x + (uint32_t)atomicAdd(a.status + kBwdDqCounter, 1);
            };
            auto publish = [&](uint32_t k, const BwdItem &w) {
                const uint32_t r = k % kItemRing;
                if (k >= kItemRing && !wait_bar(bar(C::ITEM_EMPTY + r), (k / kItemRing - 1) & 1, 2)) return false;
                tail->items[r] = w;
                ptx::mbar_arrive(bar(C::ITEM_FULL + r));
                return true;
            };
            uint32_t c = 0, kq = 0;  // steps and non-empty items so far
            BwdItem w, wn;
            w.parts = w.first = wn.parts = wn.first = 0;
            next_item(w);
            bool ok = publish(0, w);
            for (uint32_t k = 0; w.n >= 0 && ok; ++k) {
                next_item(wn);
                ok = publish(k + 1, wn);
                if (!ok) break;
                if (w.n > 0) {
                    auto load_rows = [&](uint32_t dst, const CUtensorMap *tm, uint32_t full, uint32_t empty, int code) {
                        const uint32_t rb = kq % NR;
                        if (kq >= NR && !wait_bar(bar(empty + rb), (kq / NR - 1) & 1, code)) return false;
                        ptx::mbar_expect_tx(bar(full + rb), C::kTile);
                        for (int dh = 0; dh < DH; ++dh)
                            ptx::tma_load_5d(smem_base + dst + rb * 2 * C::kTile + dh * kRowTile, tm, bar(full + rb), dh * 64,
                                             w.blk * kBwdBlk, 2 * w.hp, w.hk, w.b);
                        return true;
                    };
                    auto load_block = [&](uint32_t base, const CUtensorMap *tm, uint32_t full, uint32_t empty, uint32_t stages,
                                          int32_t j, int code) {
                        const uint32_t st = c % stages;
                        if (c >= stages && !wait_bar(bar(empty + st), (c / stages - 1) & 1, code)) return false;
                        ptx::mbar_expect_tx(bar(full + st), C::kBlkTile);
                        for (int dh = 0; dh < DH; ++dh)
                            ptx::tma_load_4d(smem_base + base + st * C::kBlkTile + dh * kKeyTile, tm, bar(full + st), dh * 64,
                                             j * kBwdBlk, w.hk, w.b);
                        return true;
                    };
                    int32_t j = a.col_idx[w.e0];
                    for (int e = 0; e < w.n && ok; ++e, ++c) {
                        const int32_t jn = e + 1 < w.n ? a.col_idx[w.e0 + e + 1] : 0;
                        if (e == 0) ok = load_rows(C::kQ, &tmQ, C::Q_FULL, C::Q_EMPTY, 3);
                        ok = ok && load_block(C::kK, &tmK, C::K_FULL, C::K_EMPTY, NK, j, 4);
                        if (e == 0) ok = ok && load_rows(C::kG, &tmG, C::G_FULL, C::G_EMPTY, 5);
                        ok = ok && load_block(C::kV, &tmV, C::V_FULL, C::V_EMPTY, NV, j, 6);
                        j = jn;
                    }
                    ++kq;
                }
                w = wn;
            }
        }
        __syncwarp();
    } else if (warp == 1 || warp == 2) {
        // -------------------------------------------------------------- tcgen05 issuers of S (warp 1) and dP (warp 2)
        const bool leader = ptx::elect_one();
        const bool is_dp = __shfl_sync(0xffffffffu, warp, 0) == 2;
        // A = Q (S) or dO (dP); B = the K or V block of the stage; both K-major.
        constexpr uint32_t idesc_s = idesc_bf16(128, 64, 0, 0);
        const uint32_t rows_full = is_dp ? C::G_FULL : C::Q_FULL, rows_empty = is_dp ? C::G_EMPTY : C::Q_EMPTY;
        const uint32_t blk_full = is_dp ? C::V_FULL : C::K_FULL, stages = is_dp ? NV : NK;
        const uint32_t out_full = is_dp ? C::DP_FULL : C::S_FULL;
        const uint32_t t_base = __shfl_sync(0xffffffffu, tmem_base + (is_dp ? C::kColDp : 0u), 0);
        uint32_t c = 0, kq = 0, st = 0, round = 0;  // step, items, the step's stage, how often the ring has come round
        bool ok = true;
        for (uint32_t k = 0; ok; ++k) {
            BwdItem w;
            ok = read_item(k, w);
            const int n = __shfl_sync(0xffffffffu, w.n, 0);
            if (!ok || n < 0) break;
            if (n == 0) continue;
            const uint32_t rb = kq % NR;
            const uint32_t a_lo = ((smem_base + rb * 2 * C::kTile + (is_dp ? C::kG : C::kQ)) >> 4) | (1u << 16);
            for (int e = 0; e < n; ++e, ++c) {
                // Three things to wait for, by three groups of lanes at a time (each wait costs some 200 clk even when it is
                // over): the block; the item's rows; the buffer (dP of two steps before is in registers; the S
                // buffer's last dS has been read).
                uint32_t b_ = blk_full + st, parity = round & 1;
                const int which = lane & 3;
                if (which == 1 && e == 0) b_ = rows_full + rb, parity = (kq / NR) & 1;
                if (which == 2 && is_dp && c >= 2) b_ = C::DP_TAKEN + (c & 1), parity = ((c >> 1) - 1) & 1;
                if (which == 2 && !is_dp && c >= 4) b_ = C::DS_FREE + (c & 3), parity = ((c >> 2) - 1) & 1;
                ok = wait_warp(bar(b_), parity, 7 + which);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                if (leader) {
                    const uint32_t b_lo = ((smem_base + (is_dp ? C::kV : C::kK) + st * C::kBlkTile) >> 4) | (1u << 16);
                    const uint32_t t_d = t_base + 64 * (is_dp ? c & 1 : c & 3);
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk)
                        ptx::umma_ss_lohi(t_d, a_lo + (((kk / 4) * kRowTile + (kk % 4) * 32) >> 4), kDescHi,
                                          b_lo + (((kk / 4) * kKeyTile + (kk % 4) * 32) >> 4), kDescHi, idesc_s,
                                          kk > 0 ? 1u : 0u);
                    ptx::umma_commit(bar(out_full + (c & 3)));
                    if (is_dp) ptx::umma_commit(bar(C::V_EMPTY + st));
                    if (e == n - 1) ptx::umma_commit(bar(rows_empty + rb));  // this warp has read the item's Q (dO) tile
                }
                __syncwarp();
                if (++st == stages) {
                    st = 0;
                    ++round;
                }
            }
            ++kq;
        }
    } else if (warp == 3) {
        // -------------------------------------------------------------- tcgen05 issuer of dQ
        const bool leader = ptx::elect_one();
        constexpr uint32_t idesc_dq = idesc_bf16(128, D, 0, 1);   // A = dS (tensor memory), B = K feature-contiguous
        const uint32_t t_base = __shfl_sync(0xffffffffu, tmem_base, 0);
        uint32_t c = 0, kq = 0;
        bool ok = true;
        for (uint32_t k = 0; ok; ++k) {
            BwdItem w;
            ok = read_item(k, w);
            const int n = __shfl_sync(0xffffffffu, w.n, 0);
            if (!ok || n < 0) break;
            if (n == 0) continue;
            for (int e = 0; e < n; ++e, ++c) {
                const uint32_t g = c & 3, st = c % NK;
                // (odd lanes: the previous item's dQ must have left tensor memory)
                const bool free = (lane & 1) && e == 0 && kq > 0;
                ok = wait_warp(bar(free ? C::DQ_FREE : C::DS_FULL + g), (free ? kq - 1 : c >> 2) & 1, free ? 11 : 10);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                if (leader) {
                    // B = the K block read feature-contiguous: 16 keys per MMA, 2048 bytes further each.
                    const uint32_t kb = ((smem_base + C::kK + st * C::kBlkTile) >> 4) | ((kKeyTile >> 4) << 16);
                    const uint32_t t_ds = t_base + 64 * g;
#pragma unroll
                    for (int kk = 0; kk < kBwdBlk / 16; ++kk)
                        ptx::umma_ts_lohi(t_base + C::kColDq, t_ds + kk * 8, kb + ((kk * 2048) >> 4), kDescHi, idesc_dq,
                                          (e > 0 || kk > 0) ? 1u : 0u);
                    ptx::umma_commit(bar(C::K_EMPTY + st));
                    ptx::umma_commit(bar(C::DS_FREE + g));
                    if (e == n - 1) ptx::umma_commit(bar(C::DQ_DONE));
                }
                __syncwarp();
            }
            ++kq;
        }
    } else if (warp < 4 + kCompWarps) {
        // -------------------------------------------------------------- compute warps
        // Warpgroup g: every fourth step.
        ptx::setmaxnreg_inc<PA_DQ_REG_COMP>();
        const uint32_t g = (uint32_t)(warp - 4) >> 2;
        const int quad = warp & 3;
        const int row = quad * 32 + lane, qrow = row & 63;
        const uint32_t t_lane = tmem_base + ((uint32_t)(quad * 32) << 16);
        const uint32_t t_s = t_lane + 64 * g, t_dp = t_lane + C::kColDp + 64 * (g & 1);
        const uint64_t scale2 = ptx::pack_f32x2(a.scale_log2, a.scale_log2);
        // An item's row data for this thread, requested one item ahead.
        float lse_n = INFINITY, delta_n = 0.f;
        int32_t lastcol_n = -1;
        auto request = [&](const BwdItem &w) {
            lse_n = INFINITY;
            delta_n = 0.f;
            lastcol_n = -1;
            if (w.n <= 0) return;
            const int head_local = 2 * w.hp + (row >> 6);
            const int64_t q = (int64_t)w.blk * kBwdBlk + qrow;
            if (head_local < a.G && q < a.N) {
                const int64_t at = ((int64_t)w.b * a.Hq + w.hk * a.G + head_local) * a.N + q;
                lse_n = a.lse[at];
                delta_n = a.delta[at];
            }
            lastcol_n = a.col_idx[w.e0 + w.n - 1];
        };
        uint32_t c = 0;  // step number at the item's start
        BwdItem w;
        bool ok = read_item(0, w);
        if (ok) request(w);
        int n = w.n, blk = w.blk;
        for (uint32_t k = 0; ok && n >= 0; ++k) {
            const float neg_lse2 = bwd_neg_lse2(lse_n);
            const uint64_t neg_lse2_2 = ptx::pack_f32x2(neg_lse2, neg_lse2), neg_delta2 = ptx::pack_f32x2(-delta_n, -delta_n);
            const bool last_is_diag = lastcol_n == blk;
            ok = read_item(k + 1, w);
            if (!ok) break;
            request(w);
            for (uint32_t e = (g - c) & 3; e < (uint32_t)n; e += 4) {
                const uint32_t phase = ((c + e) >> 2) & 1;
                uint32_t dp[64];
                ok = wait_warp(bar(C::DP_FULL + g), phase, 13);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                ptx::tmem_ld32(t_dp, *reinterpret_cast<uint32_t(*)[32]>(&dp[0]));
                ptx::tmem_ld32(t_dp + 32, *reinterpret_cast<uint32_t(*)[32]>(&dp[32]));
                ptx::tmem_wait_ld();
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(bar(C::DP_TAKEN + (g & 1)));
                ok = wait_warp(bar(C::S_FULL + g), phase, 12);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                // Algorithm 1's causal term acts inside the diagonal pair only (the row's last block).
                const bool diag = last_is_diag && (int)e == n - 1;
#pragma unroll
                for (int ch = 0; ch < 4; ++ch) {
                    uint32_t sv[16], pk[8];
                    ptx::tmem_ld16(t_s + 16 * ch, sv);
                    ptx::tmem_wait_ld();
                    if (diag) {
#pragma unroll
                        for (int x = 0; x < 16; ++x)
                            if (16 * ch + x > qrow) sv[x] = 0xff800000u;
                    }
#pragma unroll
                    for (int x = 0; x < 8; ++x)
                        pk[x] = bwd_cvt(bwd_ds(bwd_p2(sv[2 * x], sv[2 * x + 1], scale2, neg_lse2_2), dp[16 * ch + 2 * x],
                                               dp[16 * ch + 2 * x + 1], neg_delta2));
                    ptx::tmem_st8(t_s + 8 * ch, pk);  // (over S of keys that are done)
                }
                ptx::tmem_wait_st();
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(bar(C::DS_FULL + g));
            }
            c += (uint32_t)(n > 0 ? n : 0);
            n = w.n;
            blk = w.blk;
        }
    } else {
        // -------------------------------------------------------------- epilogue
        // dQ = scale x the accumulator.  A warp's 32 rows leave 32 features at a time: through a swizzled patch
        // of shared memory and a bulk tensor store each (rows beyond the sequence are clipped by the tensor
        // map).  (Plain stores moved 10 B/clk out of the SM: 7000 clk an item, during which the accumulator, or
        // 128 registers a thread, was held.)
        ptx::setmaxnreg_dec<PA_DQ_REG_EPI>();
        const int quad = warp & 3;
        const int row = quad * 32 + lane, qrow = row & 63;
        const uint32_t t_lane = tmem_base + ((uint32_t)(quad * 32) << 16);
        const uint32_t patch = smem_base + C::kOut + (uint32_t)quad * 4096u + (uint32_t)lane * 128u;
        uint32_t kq = 0;
        bool ok = true;
        for (uint32_t k = 0; ok; ++k) {
            BwdItem w;
            ok = read_item(k, w);
            if (!ok || w.n < 0) break;
            const int head_local = 2 * w.hp + (row >> 6);
            const bool head_ok = head_local < a.G;
            if (w.n == 0) {  // empty row: zero gradient, no barrier traffic
                const int64_t q = (int64_t)w.blk * kBwdBlk + qrow;
                float *dst = a.dq + (((int64_t)w.b * a.N + q) * a.Hq + w.hk * a.G + head_local) * D;
                if (head_ok && q < a.N)
                    for (int x = 0; x < D; x += 4) *reinterpret_cast<float4 *>(dst + x) = make_float4(0.f, 0.f, 0.f, 0.f);
                continue;
            }
            ok = wait_warp(bar(C::DQ_DONE), kq & 1, 15);
            if (!ok) break;
            ptx::tc_fence_after_sync();
            const int32_t tok = w.blk * kBwdBlk + 32 * (quad & 1);
#pragma unroll 1
            for (int ch = 0; ch < D / 32; ++ch) {
                uint32_t acc[32];
                ptx::tmem_ld32(t_lane + C::kColDq + 32 * ch, acc);
                ptx::tmem_wait_ld();
                if (ch == D / 32 - 1) {  // tensor memory may take the next item's first dS K
                    ptx::tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(bar(C::DQ_FREE));
                }
                if (lane == 0) ptx::bulk_wait_read_all();  // the store before has read the patch
                __syncwarp();
#pragma unroll
                for (int x = 0; x < 8; ++x)
                    ptx::st_shared_v4(patch + (uint32_t)((x ^ (lane & 7)) << 4),
                                      __float_as_uint(__uint_as_float(acc[4 * x]) * a.scale),
                                      __float_as_uint(__uint_as_float(acc[4 * x + 1]) * a.scale),
                                      __float_as_uint(__uint_as_float(acc[4 * x + 2]) * a.scale),
                                      __float_as_uint(__uint_as_float(acc[4 * x + 3]) * a.scale));
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    if (head_ok && tok < a.N)
                        ptx::tma_store_4d(&tmDq, patch, 32 * ch, tok, w.hk * a.G + head_local, w.b);
                    ptx::bulk_commit_group();
                }
            }
            ++kq;
        }
        if (lane == 0) ptx::bulk_wait_all();
    }

    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == 2) {
        // After a wait that gave up, copies and tensor-core operations issued before it may still be
        // in flight: they finish by themselves within microseconds; a bounded two milliseconds pass
        // before the tensor memory is given back.
        if (*abort_flag) {
            const long long t0 = clock64();
            while (clock64() - t0 < 4000000ll) {
            }
        }
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(tmem_base, kTcTmemCols);
    }
    pdl_wait();  // the dK / dV kernel is over, too: what follows waits for this one only
}

// ------------------------------------------------------------------------------------- dK, dV
// Bound by how long a stage of Q and dO stays occupied: loaded, read by S and dP, and read again by the second
// products once P and dS exist.  So everything that lengthens that round is cut or overlapped: Q and dO have
// rings and barriers of their own (dO is free after dV, Q after dK), P is handed over before dS, which is computed
// while dV runs, two warpgroups share a step (32 keys each) and two more work on the next one.  head_dim 128:
// three Q stages, two of dO, one buffer for P and dS each.  head_dim 64: four stages, two P / dS buffers; a
// stage's Q and dO tiles lie side by side and are read as ONE 128-row A operand [Q | dO]^T against B = [P | dS]
// (N = 128): two quadrants of the product are dV^T and dK^T, the other two are not used, and the eight MMAs take
// 512 clk where two products of 64 accumulator rows take 768.
// An item's accumulators have two buffers and warps of their own that write them out, the compute warps walk the
// steps across the ends of items, and the next item is looked up by the epilogue's first warp while the one before
// it is computed: with the lookup (a halving search, ten dependent loads) in the producer's way and the output in
// that of the compute warps, every item began with some 8000 clk in which the tensor cores stood still, against
// 10000 to 30000 of work.
// Measured before the dQ kernel ran beside it, 28 / 4 heads: the whole backward pass at 4K tokens 154 us (160 with items one
// after the other), at 32K 1430 us at full clocks (1488); 64 features, 16 / 4 heads, 2 x 8K tokens: 234 us (269).  With it
// beside: 152, 1370 and 228 us.
template <int D>
struct DkvCfg {
    static constexpr int kDH = D / 64;
    static constexpr int kQStages = D == 128 ? 3 : 4, kGStages = D == 128 ? 2 : 4, kPBufs = D == 128 ? 1 : 2;
    static constexpr uint32_t kBlkTile = kDH * kKeyTile, kTile = kDH * kRowTile;
    static constexpr uint32_t kK = 0, kV = kBlkTile;
    static constexpr uint32_t kQ = 2 * kBlkTile;
    static constexpr uint32_t kPitch = D == 128 ? kTile : 2 * kTile;  // from stage to stage
    static constexpr uint32_t kG = D == 128 ? kQ + kQStages * kTile : kQ + kTile;
    static constexpr uint32_t kPD = kQ + (kQStages + kGStages) * kTile;  // buffer: P (128 rows x 64 keys), then dS
    static constexpr uint32_t kBars = kPD + kPBufs * 2 * kRowTile;
    static constexpr uint32_t kAlloc = kBars + kBarArea + 1024;
    static_assert(kAlloc <= 227 * 1024, "shared memory budget");
    enum : uint32_t {
        KV_FULL, KV_EMPTY,
        Q_FULL, Q_EMPTY = Q_FULL + kQStages,
        G_FULL = Q_EMPTY + kQStages, G_EMPTY = G_FULL + kGStages,
        S_FULL = G_EMPTY + kGStages, S_TAKEN = S_FULL + 2,     // [step parity]
        DP_FULL = S_TAKEN + 2, DP_TAKEN = DP_FULL + 2,
        P_FULL = DP_TAKEN + 2, DS_FULL = P_FULL + kPBufs,      // [P / dS buffer]
        P_FREE = DS_FULL + kPBufs, DS_FREE = P_FREE + 2,       // [step parity]: that step's product has read it
        ACC_FULL = DS_FREE + 2, ACC_FREE = ACC_FULL + 2,       // [item parity]: dK^T and dV^T are complete / have been read
        ITEM_FULL = ACC_FREE + 2, ITEM_EMPTY = ITEM_FULL + kItemRing, COUNT = ITEM_EMPTY + kItemRing
    };
    static_assert(COUNT * 8 <= kBarBytes, "barrier area");
    // Tensor memory columns: S at 128 b, dP at 128 b + 64 (b = step parity); accumulators at 256 + 128 (item parity):
    // dK^T, then dV^T (head_dim 128), or the product with [P | dS] (head_dim 64).
    static constexpr uint32_t kColAcc = 256;
};

template <int D>
__global__ void __launch_bounds__(kTcThreads, 1)
dkv_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmG,
           const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, const BackwardArgs a,
           const uint32_t n_items)
{
    using C = DkvCfg<D>;
    constexpr int DH = C::kDH;
    constexpr uint32_t NQ = C::kQStages, NG = C::kGStages, NP = C::kPBufs;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (smem_base - ptx::smem_u32(smem_raw));
    const uint32_t bars = smem_base + C::kBars;
    BwdTail *tail = reinterpret_cast<BwdTail *>(smem + C::kBars + kBarBytes);
    volatile int *abort_flag = &tail->abort_flag;
    auto bar = [&](uint32_t idx) { return bars + idx * 8u; };
    auto wait_bar = [&](uint32_t b_, uint32_t parity, int code) {
        return ptx::mbar_wait_bounded(b_, parity, abort_flag, a.status, code, a.wait_cycles, (int)PA_ERR_TIMEOUT);
    };
    auto wait_warp = [&](uint32_t b_, uint32_t parity, int code) {
        return __all_sync(0xffffffffu, wait_bar(b_, parity, code)) != 0;
    };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto read_item = [&](uint32_t k, BwdItem &w) {
        if (!wait_warp(bar(C::ITEM_FULL + k % kItemRing), (k / kItemRing) & 1, 31)) return false;
        w = tail->items[k % kItemRing];
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(bar(C::ITEM_EMPTY + k % kItemRing));
        return true;
    };

    if (threadIdx.x == 0) {
        ptx::mbar_init(bar(C::KV_FULL), 1);
        ptx::mbar_init(bar(C::KV_EMPTY), 2);  // one commit from each of the S and dP issuers
        for (uint32_t s = 0; s < NQ; ++s) {
            ptx::mbar_init(bar(C::Q_FULL + s), 1);
            ptx::mbar_init(bar(C::Q_EMPTY + s), 1);
        }
        for (uint32_t s = 0; s < NG; ++s) {
            ptx::mbar_init(bar(C::G_FULL + s), 1);
            ptx::mbar_init(bar(C::G_EMPTY + s), 2);  // read by dP and by dV, in either order
        }
        for (int s = 0; s < 2; ++s) {
            ptx::mbar_init(bar(C::S_FULL + s), 1);
            ptx::mbar_init(bar(C::DP_FULL + s), 1);
            ptx::mbar_init(bar(C::S_TAKEN + s), kCompWarps / 2);
            ptx::mbar_init(bar(C::DP_TAKEN + s), kCompWarps / 2);
            ptx::mbar_init(bar(C::P_FREE + s), 1);
            ptx::mbar_init(bar(C::DS_FREE + s), 1);
        }
        for (uint32_t s = 0; s < NP; ++s) {
            ptx::mbar_init(bar(C::P_FULL + s), kCompWarps / 2);
            ptx::mbar_init(bar(C::DS_FULL + s), kCompWarps / 2);
        }
        for (int s = 0; s < 2; ++s) {
            ptx::mbar_init(bar(C::ACC_FULL + s), 1);
            ptx::mbar_init(bar(C::ACC_FREE + s), 4);
        }
        for (uint32_t r = 0; r < kItemRing; ++r) {
            ptx::mbar_init(bar(C::ITEM_FULL + r), 1);
            ptx::mbar_init(bar(C::ITEM_EMPTY + r), kTcThreads / 32);
        }
        tail->abort_flag = 0;
        ptx::fence_barrier_init();
        ptx::fence_proxy_async_smem();
    }
    if (warp == 2) {
        ptx::tmem_alloc(ptx::smem_u32(&tail->tmem), kTcTmemCols);
        ptx::tmem_relinquish();
    }
    pdl_wait();  // up to here this kernel may have run beside the one before it
    say_prepared(a);
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    pdl_launch_next();
    const uint32_t tmem_base = tail->tmem;

    if (warp < 4) ptx::setmaxnreg_dec<PA_DKV_REG_CTRL>();
    if (warp == 0) {
        // -------------------------------------------------------------- TMA producer
        if (lane == 0) {
            ptx::prefetch_tensormap(&tmQ);
            ptx::prefetch_tensormap(&tmG);
            ptx::prefetch_tensormap(&tmK);
            ptx::prefetch_tensormap(&tmV);
            uint32_t c = 0;  // steps so far
            bool ok = true;
            for (uint32_t k = 0; ok; ++k) {
                const uint32_t r = k % kItemRing;
                if (!wait_bar(bar(C::ITEM_FULL + r), (k / kItemRing) & 1, 32)) break;
                const BwdItem w = tail->items[r];
                ptx::mbar_arrive(bar(C::ITEM_EMPTY + r));
                if (w.n < 0) break;
                auto load_rows = [&](uint32_t dst, const CUtensorMap *tm, uint32_t full, uint32_t empty, uint32_t stages,
                                     int32_t i, int hp, int code) {
                    const uint32_t st = c % stages;
                    if (c >= stages && !wait_bar(bar(empty + st), (c / stages - 1) & 1, code)) return false;
                    ptx::mbar_expect_tx(bar(full + st), C::kTile);
                    for (int dh = 0; dh < DH; ++dh)
                        ptx::tma_load_5d(smem_base + dst + st * C::kPitch + dh * kRowTile, tm, bar(full + st), dh * 64,
                                         i * kBwdBlk, 2 * hp, w.hk, w.b);
                    return true;
                };
                int32_t i = w.first;
                for (int x = 0; x < w.n && ok; ++x) {
                    const int32_t in = x + 1 < w.n ? a.row_idx[w.e0 + x + 1] : 0;
                    for (int hp = 0; hp < a.npairs && ok; ++hp, ++c) {
                        ok = load_rows(C::kQ, &tmQ, C::Q_FULL, C::Q_EMPTY, NQ, i, hp, 33);
                        if (ok && x == 0 && hp == 0) {
                            ok = k == 0 || wait_bar(bar(C::KV_EMPTY), (k - 1) & 1, 34);
                            if (!ok) break;
                            ptx::mbar_expect_tx(bar(C::KV_FULL), 2 * C::kBlkTile);
                            for (int dh = 0; dh < DH; ++dh) {
                                ptx::tma_load_4d(smem_base + C::kK + dh * kKeyTile, &tmK, bar(C::KV_FULL), dh * 64, w.blk * kBwdBlk,
                                                 w.hk, w.b);
                                ptx::tma_load_4d(smem_base + C::kV + dh * kKeyTile, &tmV, bar(C::KV_FULL), dh * 64, w.blk * kBwdBlk,
                                                 w.hk, w.b);
                            }
                        }
                        ok = ok && load_rows(C::kG, &tmG, C::G_FULL, C::G_EMPTY, NG, i, hp, 35);
                    }
                    i = in;
                }
            }
        }
        __syncwarp();
    } else if (warp == 1 || warp == 2) {
        // -------------------------------------------------------------- tcgen05 issuers of S (warp 1) and dP (warp 2)
        const bool leader = ptx::elect_one();
        const bool is_dp = __shfl_sync(0xffffffffu, warp, 0) == 2;
        constexpr uint32_t idesc_s = idesc_bf16(128, 64, 0, 0);    // both operands K-major
        // A = Q (S) or dO (dP) of the stage; B = the key block's K or V.
        const uint32_t b_lo = ((smem_base + (is_dp ? C::kV : C::kK)) >> 4) | (1u << 16);
        const uint32_t rows_full = is_dp ? C::G_FULL : C::Q_FULL, stages = is_dp ? NG : NQ;
        const uint32_t out_full = is_dp ? C::DP_FULL : C::S_FULL, out_taken = is_dp ? C::DP_TAKEN : C::S_TAKEN;
        const uint32_t t_base = __shfl_sync(0xffffffffu, tmem_base + (is_dp ? 64u : 0u), 0);
        uint32_t c = 0, st = 0, round = 0;  // step, its stage, how often the ring has come round
        bool ok = true;
        for (uint32_t k = 0; ok; ++k) {
            BwdItem w;
            ok = read_item(k, w);
            const int n = __shfl_sync(0xffffffffu, w.n, 0) * a.npairs;
            if (!ok || n < 0) break;
            ok = wait_warp(bar(C::KV_FULL), k & 1, 36);
            for (int e = 0; e < n && ok; ++e, ++c) {
                const uint32_t bf = c & 1;
                ok = wait_warp(bar(rows_full + st), round & 1, 37);
                if (ok && c >= 2) ok = wait_warp(bar(out_taken + bf), ((c >> 1) - 1) & 1, 38);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                if (leader) {
                    const uint32_t a_lo = ((smem_base + (is_dp ? C::kG : C::kQ) + st * C::kPitch) >> 4) | (1u << 16);
                    const uint32_t t_d = t_base + 128 * bf;
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk)
                        ptx::umma_ss_lohi(t_d, a_lo + (((kk / 4) * kRowTile + (kk % 4) * 32) >> 4), kDescHi,
                                          b_lo + (((kk / 4) * kKeyTile + (kk % 4) * 32) >> 4), kDescHi, idesc_s,
                                          kk > 0 ? 1u : 0u);
                    ptx::umma_commit(bar(out_full + bf));
                    if (is_dp) ptx::umma_commit(bar(C::G_EMPTY + st));
                    if (e == n - 1) ptx::umma_commit(bar(C::KV_EMPTY));
                }
                __syncwarp();
                if (++st == stages) {
                    st = 0;
                    ++round;
                }
            }
        }
    } else if (warp == 3) {
        // -------------------------------------------------------------- tcgen05 issuer of dV^T and dK^T
        // A = the dO (Q) tile read feature-contiguous (64-feature halves kRowTile apart), B = P (dS) read
        // key-contiguous; 16 tile rows per MMA, 2048 bytes further each.
        const bool leader = ptx::elect_one();
        constexpr uint32_t idesc_t = idesc_bf16(128, D == 128 ? 64 : 128, 1, 1);
        const uint32_t t_acc = __shfl_sync(0xffffffffu, tmem_base + C::kColAcc, 0);
        uint32_t c = 0;
        bool ok = true;
        for (uint32_t k = 0; ok; ++k) {
            BwdItem w;
            ok = read_item(k, w);
            const int n = __shfl_sync(0xffffffffu, w.n, 0) * a.npairs;
            if (!ok || n < 0) break;
            // The accumulators of the item before the previous one must have been read.
            const uint32_t t_base = t_acc + 128 * (k & 1);
            if (k >= 2) ok = wait_warp(bar(C::ACC_FREE + (k & 1)), ((k >> 1) - 1) & 1, 39);
            for (int e = 0; e < n && ok; ++e, ++c) {
                const uint32_t sq = c % NQ, sg = c % NG, pb = c % NP, pphase = (c / NP) & 1;
                const uint32_t qa = ((smem_base + C::kQ + sq * C::kPitch) >> 4) | ((kRowTile >> 4) << 16);
                const uint32_t ga = ((smem_base + C::kG + sg * C::kPitch) >> 4) | ((kRowTile >> 4) << 16);
                const uint32_t pp = ((smem_base + C::kPD + pb * 2 * kRowTile) >> 4) | ((kRowTile >> 4) << 16);
                if (D == 128) {
                    // (P needs S only, so dO may not have landed yet when it is there)
                    ok = wait_warp(bar(C::G_FULL + sg), (c / NG) & 1, 47);
                    ok = ok && wait_warp(bar(C::P_FULL + pb), pphase, 40);
                    if (!ok) break;
                    ptx::tc_fence_after_sync();
                    if (leader) {
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk)
                            ptx::umma_ss_lohi(t_base + 64, ga + ((kk * 2048) >> 4), kDescHi, pp + ((kk * 2048) >> 4), kDescHi,
                                              idesc_t, (e > 0 || kk > 0) ? 1u : 0u);
                        ptx::umma_commit(bar(C::G_EMPTY + sg));
                        ptx::umma_commit(bar(C::P_FREE + (c & 1)));
                    }
                    __syncwarp();
                }
                ok = ok && wait_warp(bar(C::DS_FULL + pb), pphase, 41);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                if (leader) {
                    const uint32_t bb = D == 128 ? pp + (kRowTile >> 4) : pp;
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)
                        ptx::umma_ss_lohi(t_base, qa + ((kk * 2048) >> 4), kDescHi, bb + ((kk * 2048) >> 4), kDescHi, idesc_t,
                                          (e > 0 || kk > 0) ? 1u : 0u);
                    ptx::umma_commit(bar(C::Q_EMPTY + sq));
                    ptx::umma_commit(bar(C::DS_FREE + (c & 1)));
                    if (D == 64) ptx::umma_commit(bar(C::G_EMPTY + sg));
                    if (e == n - 1) ptx::umma_commit(bar(C::ACC_FULL + (k & 1)));
                }
                __syncwarp();
            }
        }
    } else if (warp < 4 + kCompWarps) {
        // -------------------------------------------------------------- compute warps
        // Warpgroup wg: steps of parity wg & 1, keys 32 (wg >> 1) .. + 31.
        ptx::setmaxnreg_inc<PA_DKV_REG_COMP>();
        const int wg = (warp - 4) >> 2, quad = warp & 3, par = wg & 1, half = wg >> 1;
        const int row = quad * 32 + lane, qrow = row & 63;
        const uint32_t t_lane = tmem_base + ((uint32_t)(quad * 32) << 16);
        const uint64_t scale2 = ptx::pack_f32x2(a.scale_log2, a.scale_log2);
        // The warp walks its steps without regard to where items end.  The place (item, query block in the list, head
        // pair) is that of its next step: the query block's index is requested at the start of a step for the next
        // one and the row statistics, LSE and delta, in its middle; nothing uses a loaded value on the spot.
        BwdItem w;
        uint32_t k = 0;
        int x = 0, hp = 0;
        int32_t i_next = -1;
        float lse_n = INFINITY, delta_n = 0.f;
        bool ok = read_item(0, w);
        auto advance = [&](int steps) {
            hp += steps;
            while (hp >= a.npairs) {
                hp -= a.npairs;
                ++x;
            }
            while (ok && w.n >= 0 && x >= w.n) {
                x -= w.n;
                ok = read_item(++k, w);
            }
            i_next = ok && w.n >= 0 ? a.row_idx[w.e0 + x] : -1;
        };
        auto request = [&]() {
            lse_n = INFINITY;
            delta_n = 0.f;
            const int head_local = 2 * hp + (row >> 6);
            const int64_t q = (int64_t)i_next * kBwdBlk + qrow;
            if (i_next >= 0 && head_local < a.G && q < a.N) {
                const int64_t at = ((int64_t)w.b * a.Hq + w.hk * a.G + head_local) * a.N + q;
                lse_n = a.lse[at];
                delta_n = a.delta[at];
            }
        };
        if (ok && w.n >= 0) advance(par);
        request();
        for (uint32_t cc = (uint32_t)par; ok && w.n >= 0; cc += 2) {
            const uint32_t pb = cc % NP;
            const bool diag = i_next == w.blk;
            const float neg_lse2 = bwd_neg_lse2(lse_n);
            const uint64_t neg_lse2_2 = ptx::pack_f32x2(neg_lse2, neg_lse2), neg_delta2 = ptx::pack_f32x2(-delta_n, -delta_n);
            advance(2);
            if (!ok) break;
            uint32_t x32[32];
            uint64_t p[16];
            ok = wait_warp(bar(C::S_FULL + par), (cc >> 1) & 1, 42);
            if (!ok) break;
            ptx::tc_fence_after_sync();
            ptx::tmem_ld32(t_lane + 128 * par + 32 * half, x32);
            ptx::tmem_wait_ld();
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar(C::S_TAKEN + par));
            request();  // (in flight during this step)
            // Algorithm 1's causal term acts inside the diagonal pair only.
            bwd_p(x32, diag, qrow - 32 * half, scale2, neg_lse2_2, p);
            // The P / dS buffer was read by the products of step cc - NP.  (Their barriers alternate by step
            // parity: with one buffer a warpgroup would otherwise wait for every other phase of a barrier only,
            // whose parity cannot tell two phases ahead from none.  With head_dim 64 one product reads both.)
            if (cc >= NP) {
                ok = wait_warp(bar((D == 128 ? C::P_FREE : C::DS_FREE) + ((cc - NP) & 1)), ((cc - NP) >> 1) & 1, 43);
                if (!ok) break;
            }
            // 16-byte chunk q of tile row r sits at chunk position q ^ (r & 7) (128-byte swizzle).
            const uint32_t p_row = smem_base + C::kPD + pb * 2 * kRowTile + (uint32_t)row * 128u;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                ptx::st_shared_v4(p_row + (uint32_t)(((4 * half + q) ^ (row & 7)) << 4), bwd_cvt(p[4 * q]), bwd_cvt(p[4 * q + 1]),
                                  bwd_cvt(p[4 * q + 2]), bwd_cvt(p[4 * q + 3]));
            if (D == 128) {
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(bar(C::P_FULL + pb));
            }
            ok = wait_warp(bar(C::DP_FULL + par), (cc >> 1) & 1, 44);
            if (!ok) break;
            ptx::tc_fence_after_sync();
            ptx::tmem_ld32(t_lane + 128 * par + 64 + 32 * half, x32);
            ptx::tmem_wait_ld();
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar(C::DP_TAKEN + par));
            if (D == 128 && cc >= NP) {
                ok = wait_warp(bar(C::DS_FREE + ((cc - NP) & 1)), ((cc - NP) >> 1) & 1, 45);
                if (!ok) break;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t v[4];
#pragma unroll
                for (int y = 0; y < 4; ++y)
                    v[y] = bwd_cvt(bwd_ds(p[4 * q + y], x32[8 * q + 2 * y], x32[8 * q + 2 * y + 1], neg_delta2));
                ptx::st_shared_v4(p_row + kRowTile + (uint32_t)(((4 * half + q) ^ (row & 7)) << 4), v[0], v[1], v[2], v[3]);
            }
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar(C::DS_FULL + pb));
        }
    } else {
        // -------------------------------------------------------------- epilogue warps; the first one finds the items
        ptx::setmaxnreg_dec<PA_DKV_REG_EPI>();
        const int quad = warp & 3;
        const uint32_t t_lane = tmem_base + ((uint32_t)(quad * 32) << 16);
        // Items: chunk slots in column order (the sink block's long column first); slots without work are passed over.
        // A column's listers are read by some ten columns.  Where Q and dO of all heads do not fit half of L2, one KV
        // head of one batch entry comes after the other, so that what is read again is still there; else a slot's heads
        // come together, which leaves more of the last, short columns for the end.  (L2 of an sm_100 GPU: 126 MB.)  Whole
        // backward pass in us, heads together and one after the other, by MB of Q and dO: 54 to 67 MB equal but for
        // what two runs differ by (4K tokens, 28 heads: 163.9 and 164.9; 2 x 8K, 16 heads of 64 features: 255 and 253),
        // 117 (8K) 370 and 357, 235 (16K) 778 to 838 and 685 to 788, 268 (2 x 32K of 64 features) 1120 and 1096, 470
        // (32K) 1665 and 1640 (this kernel's DRAM reads 2.4 and 1.7 GB).
        const bool by_head = (int64_t)a.batch * a.N * a.Hq * D * 4 > (int64_t)64 << 20;
        const uint32_t heads = (uint32_t)(a.Hkv * a.batch), slots = n_items / heads;
        uint32_t it = blockIdx.x;
        auto publish_next = [&](uint32_t k) {
            const uint32_t r = k % kItemRing;
            BwdItem w = {0, -1, 0, 0, 0, 0, 0, 0};
            while (it < n_items && w.n < 0) {
                const uint32_t major = it / (by_head ? slots : heads), minor = it - major * (by_head ? slots : heads);
                const uint32_t slot = by_head ? minor : major, yz = by_head ? major : minor;
                const BackwardChunk ch = backward_chunk_by_warp(a, (int32_t)slot, lane);
                if (ch.e0 < ch.e1) {
                    w.blk = ch.j;
                    w.e0 = ch.e0;
                    w.n = ch.e1 - ch.e0;
                    w.parts = ch.parts;
                    w.b = (int32_t)(yz / (uint32_t)a.Hkv);
                    w.hk = (int32_t)(yz % (uint32_t)a.Hkv);
                    w.first = a.row_idx[w.e0];
                }
                int drawn = 0;
                if (lane == 0) drawn = atomicAdd(a.status + kBwdDkvCounter, 1);
                it = gridDim.x + (uint32_t)__shfl_sync(0xffffffffu, drawn, 0);
            }
            if (k >= kItemRing && !wait_warp(bar(C::ITEM_EMPTY + r), (k / kItemRing - 1) & 1, 34)) return -2;
            // The loop below follows KV_FULL phase by phase.  So that two of its phases are never over before this warp
            // has asked for the first (their parity would then pass for that of a phase to come), item 1 is handed out
            // once the loads of item 0 have landed, which its lookup mostly outlasts.
            if (k == 1 && !wait_warp(bar(C::KV_FULL), 0, 35)) return -2;
            if (lane == 0) {
                tail->items[r] = w;
                ptx::mbar_arrive(bar(C::ITEM_FULL + r));
            }
            return w.n;
        };
        const bool finder = warp == 4 + kCompWarps;
        int n_next = -1;  // (finder) length of item k + 1
        bool ok = true;
        if (finder && publish_next(0) >= 0) n_next = publish_next(1);
        for (uint32_t k = 0; ok; ++k) {
            BwdItem w;
            ok = read_item(k, w);
            if (!ok || w.n < 0) break;
            // Item k + 2 is looked for when the loads have got to item k + 1.
            if (finder && n_next >= 0) {
                ok = wait_warp(bar(C::KV_FULL), (k + 1) & 1, 35);
                if (!ok) break;
                n_next = publish_next(k + 2);
            }
            ok = wait_warp(bar(C::ACC_FULL + (k & 1)), (k >> 1) & 1, 46);
            if (!ok) break;
            ptx::tc_fence_after_sync();
            // A lane holds a feature and a register a key.  Quads of lanes transpose 4 x 4 among themselves, so that
            // a lane gets four features of a key: 16 bytes.  A key block of one chunk is written, the parts of others
            // are added up in memory.  (The four warps take 12000 clk for an item's 64 KB, 26000 with 4 bytes a lane
            // and 14000 with 32 keys at a time, for which the addresses find no registers.)
            const int64_t pitch = (int64_t)a.Hkv * D;
            constexpr int kChunks = D == 128 ? 8 : 4;  // of 16 accumulator columns that the warp takes
#pragma unroll 1
            for (int ch = 0; ch < kChunks; ++ch) {
                const bool is_dk = D == 128 ? ch < 4 : quad < 2;
                uint32_t acc[16];
                ptx::tmem_ld16(t_lane + C::kColAcc + 128 * (k & 1) + (D == 64 && is_dk ? 64 : 0) + 16 * ch, acc);
                ptx::tmem_wait_ld();
                if (ch == kChunks - 1) {
                    ptx::tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(bar(C::ACC_FREE + (k & 1)));
                }
                const int64_t tok0 = (int64_t)w.blk * kBwdBlk + 16 * (ch & 3) + (lane & 3);
                const int keys = a.N - tok0 < 16 ? (int)(a.N - tok0) : 16;
                float *dst = (is_dk ? a.dk : a.dv) + (((int64_t)w.b * a.N + tok0) * a.Hkv + w.hk) * D +
                             ((quad * 32 + lane) & (D - 4));
                const float f = is_dk ? a.scale : 1.0f;
                float *at[4];
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    transpose_quad(acc[4 * x], acc[4 * x + 1], acc[4 * x + 2], acc[4 * x + 3], lane);
                    at[x] = dst + 4 * x * pitch;
                }
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const float4 v = make_float4(__uint_as_float(acc[4 * x]) * f, __uint_as_float(acc[4 * x + 1]) * f,
                                                 __uint_as_float(acc[4 * x + 2]) * f, __uint_as_float(acc[4 * x + 3]) * f);
                    if (4 * x < keys) {
                        if (w.parts == 1) *reinterpret_cast<float4 *>(at[x]) = v;
                        else ptx::red_add_v4(at[x], v);
                    }
                }
            }
        }
    }

    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == 2) {
        if (*abort_flag) {
            const long long t0 = clock64();
            while (clock64() - t0 < 4000000ll) {
            }
        }
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(tmem_base, kTcTmemCols);
    }
}

// dK = dV = 0 for key blocks that are added up from several chunks, or that nobody lists (where the preparation has not
// cleared everything).
constexpr int kClearThreads = 256;
__global__ void __launch_bounds__(kClearThreads) backward_clear_kernel(const BackwardArgs a, const int32_t D)
{
    pdl_wait();
    const int64_t per_token = (int64_t)a.Hkv * D / 4;
    for (int32_t j = blockIdx.x; j < a.nqb; j += gridDim.x) {
        const int32_t cnt = a.col_ptr[j + 1] - a.col_ptr[j];
        if (cnt > 0 && cnt <= a.chunk) continue;
        const int64_t tok0 = (int64_t)j * kBwdBlk, toks = a.N - tok0 < kBwdBlk ? a.N - tok0 : kBwdBlk;
        for (int32_t b = 0; b < a.batch; ++b) {
            float4 *zk = reinterpret_cast<float4 *>(a.dk) + (b * a.N + tok0) * per_token;
            float4 *zv = reinterpret_cast<float4 *>(a.dv) + (b * a.N + tok0) * per_token;
            for (int64_t x = blockIdx.y * kClearThreads + threadIdx.x; x < toks * per_token; x += gridDim.y * kClearThreads)
                zk[x] = zv[x] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
}

// ---------------------------------------------------------------------------------- host side
template <int D>
static pa_status launch_tc(const BackwardArgs &a, const pa_prefill_params *p, int64_t nnz, int device, int sms, cudaStream_t st)
{
    // Tensor maps (cached per buffer and shape): a Q or dO box holds the two heads of a tile, a K or V box one head.
    // The last tile of a group with an odd number of heads gets zeros for the second: both products of a tile sum over its
    // rows, so that whatever another group's head holds there (infinities, NaN) would reach this group's dK and dV.
    CUtensorMap tmQ, tmG, tmK, tmV, tmDq;
    auto map_of = [&](const void *base, int heads, const pa_strides &s, int box_heads, int group, const char *what,
                      CUtensorMap *m) {
        const TensorMapKey key = {base,  p->seq_len, s.seq,     s.head,  s.batch, device, D,
                                  heads, p->batch,   box_heads, kBwdBlk, 0,       group};
        return get_tensor_map(key, what, m);
    };
    if (pa_status s = map_of(a.q, a.Hq, p->q, 2, a.G, "q", &tmQ)) return s;
    if (pa_status s = map_of(a.d_o, a.Hq, p->o, 2, a.G, "d_o", &tmG)) return s;
    if (pa_status s = map_of(a.k, a.Hkv, p->k, 1, 0, "k", &tmK)) return s;
    if (pa_status s = map_of(a.v, a.Hkv, p->v, 1, 0, "v", &tmV)) return s;
    const int64_t dq_seq = (int64_t)a.Hq * D;
    const TensorMapKey out = {a.dq, p->seq_len, dq_seq, D, a.N * dq_seq, device, D, a.Hq, p->batch, 1, 32, 1};
    if (pa_status s = get_tensor_map(out, "dq", &tmDq)) return s;
    if (pa_status s = device_once(device, D == 128 ? ONCE_BACKWARD_TC_ATTR : ONCE_BACKWARD_TC_ATTR_64, [] {
            constexpr cudaFuncAttribute kSmem = cudaFuncAttributeMaxDynamicSharedMemorySize;
            return first_error(cudaFuncSetAttribute(dq_kernel<D>, kSmem, (int)DqCfg<D>::kAlloc),
                               cudaFuncSetAttribute(dkv_kernel<D>, kSmem, (int)DkvCfg<D>::kAlloc));
        }))
        return s;
    const int64_t dq_items = (int64_t)a.nqb * a.Hkv * a.npairs * a.batch;
    const int64_t dkv_items = (nnz / a.chunk + a.nqb) * a.Hkv * a.batch;  // (chunk slots, some of them empty)
    if (dq_items > (int64_t)0x3fffffff || dkv_items > (int64_t)0x3fffffff)
        return fail(PA_ERR_SHAPE, "too many work items (%lld, %lld)", (long long)dq_items, (long long)dkv_items);
    if (!a.prezero)
        PA_CUDA_OK(launch_pdl(backward_clear_kernel, dim3((unsigned)(a.nqb < sms ? a.nqb : sms), 8), kClearThreads, 0, st, a,
                              (int32_t)D));
    PA_CUDA_OK(launch_pdl(dkv_kernel<D>, dim3((unsigned)(dkv_items < sms ? dkv_items : sms)), kTcThreads, DkvCfg<D>::kAlloc, st,
                          tmQ, tmG, tmK, tmV, a, (uint32_t)dkv_items));
    PA_CUDA_OK(launch_pdl(dq_kernel<D>, dim3((unsigned)(dq_items < sms ? dq_items : sms)), kTcThreads, DqCfg<D>::kAlloc, st, tmQ,
                          tmG, tmK, tmV, tmDq, a, (uint32_t)dq_items));
    return PA_OK;
}

pa_status launch_backward_sm100(const BackwardArgs &args, const pa_prefill_params *p, int64_t nnz, int device, int sms,
                                cudaStream_t st)
{
    BackwardArgs a = args;
    const long long wait_cycles = wait_limit_cycles();
    a.wait_cycles = wait_cycles > 0 ? wait_cycles : kBwdWaitCycles;
    return p->head_dim == 128 ? launch_tc<128>(a, p, nnz, device, sms, st) : launch_tc<64>(a, p, nnz, device, sms, st);
}

}  // namespace pa
