// Backward pass of the block-sparse attention (derivatives of Eq. (1), Section 3.1, under the
// key-block lists of Algorithm 1, Section 3.3) on the sm_100a tensor cores, head_dim 64 and 128.
//
// Two kernels (dK / dV: head_dim 128 only).  The dQ kernel's warps:
//   warp 0       TMA producer (bf16 tiles, 128-byte swizzle, into rings of shared-memory stages); it also draws
//                the CTA's next work item from a counter in memory and hands it to the other warps through a
//                small ring in shared memory
//   warp 1       tcgen05 issuer of S (one elected lane)
//   warp 2       tensor-memory allocation, issuer of dP
//   warp 3       issuer of the second products
//   warps 4-19   four compute warpgroups
//   warps 20-23  epilogue: the finished dQ out of tensor memory and out to global memory
// The dK / dV kernel has the same warps 0-3 (without items: a CTA has one), and two compute warpgroups (warps
// 4-11) which take alternate steps.
// A step is one query block and one (dK / dV kernel) or two (dQ kernel) of its key blocks for a pair of query
// heads stacked on the 64 tokens of the query block: a 128-row tile, as in the forward kernel.  Per step the
// tensor cores produce S = Q K^T and dP = dO V^T (fp32, tensor memory); the compute warps (thread = tile row =
// TMEM lane) turn them into P = exp2(S scale log2e - LSE log2e) and dS = P (dP - delta), rounded
// to bf16; the second products accumulate in tensor memory.
//
//   dq_kernel   an item is a (query block, head pair): walks the row's key blocks two at a time; dS goes back
//               into tensor memory as the A operand of dQ += dS K (128 x D accumulator)
//   dkv_kernel  one CTA per (chunk of a key block's listing query blocks, KV head): walks the chunk for every
//               head pair of the group; P and dS go to shared memory as the B operands of dV^T += dO^T P and
//               dK^T += Q^T dS (feature x key accumulators: the A operands are the dO and Q tiles read
//               feature-major)
//
// Every barrier wait is bounded; a wait that runs out records PA_ERR_TIMEOUT in the status block,
// raises a CTA-wide abort flag, every role leaves its loop and the CTA ends after a bounded pause.
#include <cuda.h>
#include <cuda_bf16.h>
#include <math.h>

#include "backward.cuh"
#include "sm100_ptx.cuh"
#include "tensor_map.cuh"

// Registers per thread by role.  A warpgroup asking for more than the pool holds would wait for ever: the dK / dV
// kernel starts 384 threads x 168, the dQ kernel 768 x 80.
#define PA_BWD_REG_CTRL 56
#define PA_BWD_REG_COMP 216
static_assert(4 * PA_BWD_REG_CTRL + 8 * PA_BWD_REG_COMP <= 12 * 168, "register split exceeds the CTA's registers");
#define PA_DQ_REG_CTRL 48
#define PA_DQ_REG_COMP 96
#define PA_DQ_REG_EPI 48
static_assert(4 * PA_DQ_REG_CTRL + 16 * PA_DQ_REG_COMP + 4 * PA_DQ_REG_EPI <= 24 * 80, "register split exceeds the CTA's registers");

namespace pa {

constexpr int kTcThreads = 384;
constexpr int kDqThreads = 768;
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
// its row or chunk lists, from e0 on (negative: there are no more items); parts: chunks of the key block.
struct __align__(16) BwdItem {
    int32_t blk, n, e0, hk, b, hp, parts, pad;
};
struct BwdTail {
    BwdItem items[kItemRing];
    uint32_t tmem;
    int abort_flag;
};
static_assert(kBarBytes + sizeof(BwdTail) <= kBarArea, "barrier area");

// P = exp2(S scale - lse2) of 32 keys, as packed pairs; keys beyond `lim` (causal term of the diagonal pair) are 0.
__device__ __forceinline__ void bwd_p(uint32_t (&s)[32], bool diag, int lim, uint64_t scale2, uint64_t neg_lse2,
                                      uint64_t (&p)[16])
{
    if (diag) {
#pragma unroll
        for (int x = 0; x < 32; ++x)
            if (x > lim) s[x] = 0xff800000u;
    }
#pragma unroll
    for (int x = 0; x < 16; ++x) {
        const uint64_t y2 = ptx::fma_f32x2(ptx::pack_f32x2(__uint_as_float(s[2 * x]), __uint_as_float(s[2 * x + 1])), scale2,
                                           neg_lse2);
        float y0, y1;
        ptx::unpack_f32x2(y2, y0, y1);
        p[x] = ptx::pack_f32x2(ptx::ex2(y0), ptx::ex2(y1));
    }
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
// -LSE in base 2; a row without weights (beyond the sequence, padding head, empty row) gets -inf: P = 0.
__device__ __forceinline__ float bwd_neg_lse2(float lse)
{
    return (lse == -INFINITY || lse == INFINITY) ? -INFINITY : -lse * 1.4426950408889634f;
}

// ------------------------------------------------------------------------------------- dQ
// Two key blocks a step: S and dP are 128 x 128 MMAs (N = 64 reads A again for half the work: 48 clk instead of
// 32 for 64 keys), and the fixed cost of a step, barrier round trips and the warps' loads and stores, is paid
// once for both.  A row of odd length ends on a step of one block, for which the second block's compute warps
// only keep the barriers going.  S and dP have one buffer each: the warps take them into registers at once, 32
// keys a thread, and the next step's products run beside the arithmetic.  Q and dO have one buffer each as well:
// the next item's tiles arrive while the last step is computed and its dQ product runs.
// Measured, 28 / 4 heads at 32K tokens: 586 us, where steps of one block with two S and dP buffers took 661; 64
// features, 16 / 4 heads, 2 x 8K tokens: 109 us, where the warp-level MMA kernel took 218.
template <int D>
struct DqCfg {
    static constexpr int kDH = D / 64;
    static constexpr int kStages = D == 128 ? 2 : 4;         // K and V rings, each of two blocks
    static constexpr uint32_t kTile = kDH * kRowTile;        // Q, dO, and a pair of K or V blocks
    static constexpr uint32_t kQ = 0, kG = kTile;
    static constexpr uint32_t kK = 2 * kTile, kV = kK + kStages * kTile;
    static constexpr uint32_t kOut = kV + kStages * kTile;   // per epilogue warp two patches of 32 rows x 32 fp32
    static constexpr uint32_t kBars = kOut + 4 * 2 * 4096;
    static constexpr uint32_t kAlloc = kBars + kBarArea + 1024;
    static_assert(kAlloc <= 227 * 1024, "shared memory budget");
    enum : uint32_t {
        Q_FULL, Q_EMPTY, G_FULL, G_EMPTY,
        K_FULL, K_EMPTY = K_FULL + kStages,
        V_FULL = K_EMPTY + kStages, V_EMPTY = V_FULL + kStages,
        S_FULL = V_EMPTY + kStages, S_TAKEN, DP_FULL, DP_TAKEN,
        DS_FULL, DS_FREE = DS_FULL + 2,      // [step parity]
        DQ_DONE = DS_FREE + 2,               // the item's last dQ += dS K has completed
        DQ_FREE,                             // the epilogue warps have read dQ out of tensor memory
        ITEM_FULL, ITEM_EMPTY = ITEM_FULL + kItemRing, COUNT = ITEM_EMPTY + kItemRing
    };
    static_assert(COUNT * 8 <= kBarBytes, "barrier area");
    // Tensor memory columns: S, dP, dS (bf16 pairs, two buffers), dQ.
    static constexpr uint32_t kColDp = 128, kColDs = 256, kColDq = 384;
};

template <int D>
__global__ void __launch_bounds__(kDqThreads, 1)
dq_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmG,
          const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
          const __grid_constant__ CUtensorMap tmDq, const BackwardArgs a, const uint32_t n_items)
{
    using C = DqCfg<D>;
    constexpr int DH = C::kDH;
    constexpr uint32_t kStages = C::kStages;
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
        ptx::mbar_init(bar(C::Q_FULL), 1);
        ptx::mbar_init(bar(C::Q_EMPTY), 1);
        ptx::mbar_init(bar(C::G_FULL), 1);
        ptx::mbar_init(bar(C::G_EMPTY), 1);
        for (uint32_t s = 0; s < kStages; ++s) {
            ptx::mbar_init(bar(C::K_FULL + s), 1);
            ptx::mbar_init(bar(C::K_EMPTY + s), 1);
            ptx::mbar_init(bar(C::V_FULL + s), 1);
            ptx::mbar_init(bar(C::V_EMPTY + s), 1);
        }
        ptx::mbar_init(bar(C::S_FULL), 1);
        ptx::mbar_init(bar(C::DP_FULL), 1);
        ptx::mbar_init(bar(C::S_TAKEN), kCompWarps);
        ptx::mbar_init(bar(C::DP_TAKEN), kCompWarps);
        for (int s = 0; s < 2; ++s) {
            ptx::mbar_init(bar(C::DS_FULL + s), kCompWarps);
            ptx::mbar_init(bar(C::DS_FREE + s), 1);
        }
        ptx::mbar_init(bar(C::DQ_DONE), 1);
        ptx::mbar_init(bar(C::DQ_FREE), 4);
        for (uint32_t r = 0; r < kItemRing; ++r) {
            ptx::mbar_init(bar(C::ITEM_FULL + r), 1);
            ptx::mbar_init(bar(C::ITEM_EMPTY + r), kDqThreads / 32 - 1);
        }
        tail->abort_flag = 0;
        ptx::fence_barrier_init();
        ptx::fence_proxy_async_smem();
    }
    if (warp == 2) {
        ptx::tmem_alloc(ptx::smem_u32(&tail->tmem), kTcTmemCols);
        ptx::tmem_relinquish();
    }
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
                w.e0 = __ldg(a.row_ptr + w.blk);
                w.n = __ldg(a.row_ptr + w.blk + 1) - w.e0;
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
            w.parts = w.pad = wn.parts = wn.pad = 0;
            next_item(w);
            bool ok = publish(0, w);
            for (uint32_t k = 0; w.n >= 0 && ok; ++k) {
                next_item(wn);
                ok = publish(k + 1, wn);
                if (!ok) break;
                if (w.n > 0) {
                    const int h0 = w.hk * a.G + 2 * w.hp;
                    auto load_rows = [&](uint32_t dst, const CUtensorMap *tm, uint32_t full, uint32_t empty, int code) {
                        if (kq >= 1 && !wait_bar(bar(empty), (kq - 1) & 1, code)) return false;
                        ptx::mbar_expect_tx(bar(full), C::kTile);
                        for (int dh = 0; dh < DH; ++dh)
                            ptx::tma_load_4d(smem_base + dst + dh * kRowTile, tm, bar(full), dh * 64, w.blk * kBwdBlk, h0, w.b);
                        return true;
                    };
                    auto load_pair = [&](uint32_t base, const CUtensorMap *tm, uint32_t full, uint32_t empty, int32_t j0, int32_t j1,
                                         int code) {
                        const uint32_t st = c % kStages;
                        if (c >= kStages && !wait_bar(bar(empty + st), (c / kStages - 1) & 1, code)) return false;
                        const uint32_t dst = smem_base + base + st * C::kTile;
                        ptx::mbar_expect_tx(bar(full + st), (j1 >= 0 ? 2u : 1u) * DH * kKeyTile);
                        for (int dh = 0; dh < DH; ++dh) {
                            ptx::tma_load_4d(dst + dh * kRowTile, tm, bar(full + st), dh * 64, j0 * kBwdBlk, w.hk, w.b);
                            if (j1 >= 0)
                                ptx::tma_load_4d(dst + dh * kRowTile + kKeyTile, tm, bar(full + st), dh * 64, j1 * kBwdBlk, w.hk, w.b);
                        }
                        return true;
                    };
                    int32_t j0 = __ldg(a.col_idx + w.e0), j1 = w.n > 1 ? __ldg(a.col_idx + w.e0 + 1) : -1;
                    for (int e = 0; e < w.n && ok; e += 2, ++c) {
                        const int32_t j0n = e + 2 < w.n ? __ldg(a.col_idx + w.e0 + e + 2) : 0;
                        const int32_t j1n = e + 3 < w.n ? __ldg(a.col_idx + w.e0 + e + 3) : -1;
                        if (e == 0) ok = load_rows(C::kQ, &tmQ, C::Q_FULL, C::Q_EMPTY, 3);
                        ok = ok && load_pair(C::kK, &tmK, C::K_FULL, C::K_EMPTY, j0, j1, 4);
                        if (e == 0) ok = ok && load_rows(C::kG, &tmG, C::G_FULL, C::G_EMPTY, 5);
                        ok = ok && load_pair(C::kV, &tmV, C::V_FULL, C::V_EMPTY, j0, j1, 6);
                        j0 = j0n;
                        j1 = j1n;
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
        // A = Q (S) or dO (dP); B = the K or V blocks of the stage; both K-major.
        const uint32_t a_lo = ((smem_base + (is_dp ? C::kG : C::kQ)) >> 4) | (1u << 16);
        const uint32_t rows_full = is_dp ? C::G_FULL : C::Q_FULL, rows_empty = is_dp ? C::G_EMPTY : C::Q_EMPTY;
        const uint32_t blk_full = is_dp ? C::V_FULL : C::K_FULL;
        const uint32_t out_full = is_dp ? C::DP_FULL : C::S_FULL, out_taken = is_dp ? C::DP_TAKEN : C::S_TAKEN;
        const uint32_t t_d = __shfl_sync(0xffffffffu, tmem_base + (is_dp ? C::kColDp : 0u), 0);
        uint32_t c = 0, kq = 0;
        bool ok = true;
        for (uint32_t k = 0; ok; ++k) {
            BwdItem w;
            ok = read_item(k, w);
            const int n = __shfl_sync(0xffffffffu, w.n, 0);
            if (!ok || n < 0) break;
            if (n == 0) continue;
            for (int e = 0; e < n; e += 2, ++c) {
                const uint32_t st = c % kStages;
                if (e == 0) ok = wait_warp(bar(rows_full), kq & 1, 7);
                ok = ok && wait_warp(bar(blk_full + st), (c / kStages) & 1, 8);
                if (c >= 1) ok = ok && wait_warp(bar(out_taken), (c - 1) & 1, 9);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                if (leader) {
                    const uint32_t b_lo = ((smem_base + (is_dp ? C::kV : C::kK) + st * C::kTile) >> 4) | (1u << 16);
                    const uint32_t idesc = e + 1 < n ? idesc_bf16(128, 128, 0, 0) : idesc_bf16(128, 64, 0, 0);
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk)
                        ptx::umma_ss_lohi(t_d, a_lo + (((kk / 4) * kRowTile + (kk % 4) * 32) >> 4), kDescHi,
                                          b_lo + (((kk / 4) * kRowTile + (kk % 4) * 32) >> 4), kDescHi, idesc, kk > 0 ? 1u : 0u);
                    ptx::umma_commit(bar(out_full));
                    if (is_dp) ptx::umma_commit(bar(C::V_EMPTY + st));
                    if (e + 2 >= n) ptx::umma_commit(bar(rows_empty));  // this warp has read the item's Q (dO) tile
                }
                __syncwarp();
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
            for (int e = 0; e < n; e += 2, ++c) {
                const uint32_t bf = c & 1, st = c % kStages;
                ok = wait_warp(bar(C::DS_FULL + bf), (c >> 1) & 1, 10);
                // The previous item's dQ must have left tensor memory.
                if (ok && e == 0 && kq > 0) ok = wait_warp(bar(C::DQ_FREE), (kq - 1) & 1, 11);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                if (leader) {
                    // B = the K blocks read feature-contiguous: 16 keys per MMA, 2048 bytes further each.
                    const uint32_t kb = ((smem_base + C::kK + st * C::kTile) >> 4) | ((kRowTile >> 4) << 16);
                    const uint32_t t_ds = t_base + C::kColDs + 64 * bf;
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)
                        if (kk < 4 || e + 1 < n)
                            ptx::umma_ts_lohi(t_base + C::kColDq, t_ds + kk * 8, kb + ((kk * 2048) >> 4), kDescHi, idesc_dq,
                                              (e > 0 || kk > 0) ? 1u : 0u);
                    ptx::umma_commit(bar(C::K_EMPTY + st));
                    ptx::umma_commit(bar(C::DS_FREE + bf));
                    if (e + 2 >= n) ptx::umma_commit(bar(C::DQ_DONE));
                }
                __syncwarp();
            }
            ++kq;
        }
    } else if (warp < 4 + kCompWarps) {
        // -------------------------------------------------------------- compute warps
        // Warpgroup wg: keys 32 wg .. 32 wg + 31 of the step's 128.
        ptx::setmaxnreg_inc<PA_DQ_REG_COMP>();
        const int wg = (warp - 4) >> 2, quad = warp & 3, blk = wg >> 1;
        const int row = quad * 32 + lane, qrow = row & 63;
        const uint32_t t_lane = tmem_base + ((uint32_t)(quad * 32) << 16);
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
                lse_n = __ldg(a.lse + at);
                delta_n = __ldg(a.delta + at);
            }
            lastcol_n = __ldg(a.col_idx + w.e0 + w.n - 1);
        };
        uint32_t c = 0;
        BwdItem w, wn;
        bool ok = read_item(0, w);
        if (ok) request(w);
        for (uint32_t k = 0; ok && w.n >= 0; ++k) {
            const float neg_lse2 = bwd_neg_lse2(lse_n);
            const uint64_t neg_lse2_2 = ptx::pack_f32x2(neg_lse2, neg_lse2), neg_delta2 = ptx::pack_f32x2(-delta_n, -delta_n);
            const bool last_is_diag = lastcol_n == w.blk;
            ok = read_item(k + 1, wn);
            if (!ok) break;
            request(wn);
            for (int e = 0; e < w.n; e += 2, ++c) {
                const bool active = e + blk < w.n;
                uint32_t x32[32];
                uint64_t p[16];
                ok = wait_warp(bar(C::S_FULL), c & 1, 12);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                if (active) {
                    ptx::tmem_ld32(t_lane + 32 * wg, x32);
                    ptx::tmem_wait_ld();
                }
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(bar(C::S_TAKEN));
                // Algorithm 1's causal term acts inside the diagonal pair only (the row's last block).
                if (active)
                    bwd_p(x32, last_is_diag && e + blk == w.n - 1, qrow - 32 * (wg & 1), scale2, neg_lse2_2, p);
                ok = wait_warp(bar(C::DP_FULL), c & 1, 13);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                if (active) {
                    ptx::tmem_ld32(t_lane + C::kColDp + 32 * wg, x32);
                    ptx::tmem_wait_ld();
                }
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(bar(C::DP_TAKEN));
                if (c >= 2) {
                    ok = wait_warp(bar(C::DS_FREE + (c & 1)), ((c >> 1) - 1) & 1, 14);
                    if (!ok) break;
                }
                if (active) {
                    uint32_t pk[16];
#pragma unroll
                    for (int x = 0; x < 16; ++x) pk[x] = bwd_cvt(bwd_ds(p[x], x32[2 * x], x32[2 * x + 1], neg_delta2));
                    ptx::tmem_st16(t_lane + C::kColDs + 64 * (c & 1) + 16 * wg, pk);
                    ptx::tmem_wait_st();
                }
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(bar(C::DS_FULL + (c & 1)));
            }
            w = wn;
        }
    } else {
        // -------------------------------------------------------------- epilogue
        // dQ = scale x the accumulator.  A warp's 32 rows leave 32 features at a time: through a swizzled patch of
        // shared memory and a bulk tensor store each (rows beyond the sequence are clipped by the tensor map), two
        // patches in turn.  (Plain stores moved 10 B/clk out of the SM: 7000 clk an item, during which the
        // accumulator, or 128 registers a thread, was held.)
        ptx::setmaxnreg_dec<PA_DQ_REG_EPI>();
        const int quad = warp & 3;
        const int row = quad * 32 + lane, qrow = row & 63;
        const uint32_t t_lane = tmem_base + ((uint32_t)(quad * 32) << 16);
        const uint32_t patch = smem_base + C::kOut + (uint32_t)quad * 8192u + (uint32_t)lane * 128u;
        uint32_t kq = 0, np = 0;
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
            for (int ch = 0; ch < D / 32; ++ch, ++np) {
                uint32_t acc[32];
                ptx::tmem_ld32(t_lane + C::kColDq + 32 * ch, acc);
                ptx::tmem_wait_ld();
                if (ch == D / 32 - 1) {  // tensor memory may take the next item's first dS K
                    ptx::tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(bar(C::DQ_FREE));
                }
                if (lane == 0) ptx::bulk_wait_read<1>();  // the store before last has read this patch
                __syncwarp();
                const uint32_t buf = 4096u * (np & 1), dst = patch + buf;
#pragma unroll
                for (int x = 0; x < 8; ++x)
                    ptx::st_shared_v4(dst + (uint32_t)((x ^ (lane & 7)) << 4), __float_as_uint(__uint_as_float(acc[4 * x]) * a.scale),
                                      __float_as_uint(__uint_as_float(acc[4 * x + 1]) * a.scale),
                                      __float_as_uint(__uint_as_float(acc[4 * x + 2]) * a.scale),
                                      __float_as_uint(__uint_as_float(acc[4 * x + 3]) * a.scale));
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    if (head_ok && tok < a.N)
                        ptx::tma_store_4d(&tmDq, dst, 32 * ch, tok, w.hk * a.G + head_local, w.b);
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
}

// ------------------------------------------------------------------------------------- dK, dV
struct DkvSmem {
    static constexpr uint32_t kK = 0;                        // two halves of 64 keys x 128 B
    static constexpr uint32_t kV = kK + 2 * kKeyTile;
    static constexpr uint32_t kQG = kV + 2 * kKeyTile;       // stage: Q (two halves of 128 rows x 128 B), then dO
    static constexpr uint32_t kStage = 4 * kRowTile;
    static constexpr uint32_t kPD = kQG + 2 * kStage;        // buffer: P (128 rows x 64 keys), then dS
    static constexpr uint32_t kBuf = 2 * kRowTile;
    static constexpr uint32_t kBars = kPD + 2 * kBuf;
    static constexpr uint32_t kAlloc = kBars + 512 + 1024;
    static_assert(kAlloc <= 227 * 1024, "shared memory budget");
};
enum : uint32_t {
    KV_KV_FULL = 0,
    KV_QG_FULL = 1, KV_QG_EMPTY = 3,  // [stage]
    KV_SD_FULL = 5,                   // [buffer]: S and dP of a step are in tensor memory
    KV_S_TAKEN = 7,                   // [buffer]: the group has them in registers
    KV_PD_FULL = 9,                   // [buffer]: P and dS are in shared memory
    KV_DONE = 11,
    KV_BAR_COUNT = 12
};

__global__ void __launch_bounds__(kTcThreads, 1)
dkv_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmG,
           const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, const BackwardArgs a)
{
    constexpr int D = 128;
    using SM = DkvSmem;
    const BackwardChunk chunk = backward_chunk_at(a, (int32_t)blockIdx.x);
    const int32_t j = chunk.j, e0 = chunk.e0, e1 = chunk.e1;
    if (e0 >= e1) return;  // (the grid is an upper bound on the number of chunks)
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (smem_base - ptx::smem_u32(smem_raw));
    const uint32_t bars = smem_base + SM::kBars;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + SM::kBars + KV_BAR_COUNT * 8);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + SM::kBars + KV_BAR_COUNT * 8 + 8);
    auto bar = [&](uint32_t idx) { return bars + idx * 8u; };
    auto wait_bar = [&](uint32_t b_, uint32_t parity, int code) {
        return ptx::mbar_wait_bounded(b_, parity, abort_flag, a.status, code, a.wait_cycles, (int)PA_ERR_TIMEOUT);
    };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int hk = blockIdx.y, b = blockIdx.z;
    const int n = (e1 - e0) * a.npairs;  // steps: listing query blocks x head pairs (pairs fastest); at least one

    if (threadIdx.x == 0) {
        ptx::mbar_init(bar(KV_KV_FULL), 1);
        for (int s = 0; s < 2; ++s) {
            ptx::mbar_init(bar(KV_QG_FULL + s), 1);
            ptx::mbar_init(bar(KV_QG_EMPTY + s), 1);
            ptx::mbar_init(bar(KV_SD_FULL + s), 2);  // one commit from each of the S and dP issuers
            ptx::mbar_init(bar(KV_S_TAKEN + s), 4);
            ptx::mbar_init(bar(KV_PD_FULL + s), 4);
        }
        ptx::mbar_init(bar(KV_DONE), 1);
        *abort_flag = 0;
        ptx::fence_barrier_init();
        ptx::fence_proxy_async_smem();
    }
    if (warp == 2) {
        ptx::tmem_alloc(ptx::smem_u32(tmem_slot), kTcTmemCols);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    // Tensor memory columns: buffer b: S at 128 b, dP at 128 b + 64; dK^T at 256, dV^T at 320 (64 keys each).
    constexpr uint32_t kColDk = 256, kColDv = 320;

    if (warp < 4) ptx::setmaxnreg_dec<PA_BWD_REG_CTRL>();
    if (warp == 0) {
        // -------------------------------------------------------------- TMA producer
        if (lane == 0) {
            ptx::prefetch_tensormap(&tmQ);
            ptx::prefetch_tensormap(&tmG);
            ptx::prefetch_tensormap(&tmK);
            ptx::prefetch_tensormap(&tmV);
            ptx::mbar_expect_tx(bar(KV_KV_FULL), 4 * kKeyTile);
            for (int dh = 0; dh < 2; ++dh) {
                ptx::tma_load_4d(smem_base + SM::kK + dh * kKeyTile, &tmK, bar(KV_KV_FULL), dh * 64, j * kBwdBlk, hk, b);
                ptx::tma_load_4d(smem_base + SM::kV + dh * kKeyTile, &tmV, bar(KV_KV_FULL), dh * 64, j * kBwdBlk, hk, b);
            }
            int32_t i = 0;
            for (int e = 0, hp = 0; e < n; ++e) {
                if (hp == 0) i = __ldg(a.row_idx + e0 + e / a.npairs);
                const uint32_t st = e & 1;
                if (e >= 2 && !wait_bar(bar(KV_QG_EMPTY + st), ((e >> 1) - 1) & 1, 2)) break;
                ptx::mbar_expect_tx(bar(KV_QG_FULL + st), SM::kStage);
                const uint32_t dst = smem_base + SM::kQG + st * SM::kStage;
                const int h0 = hk * a.G + 2 * hp;
                for (int dh = 0; dh < 2; ++dh) {
                    ptx::tma_load_4d(dst + dh * kRowTile, &tmQ, bar(KV_QG_FULL + st), dh * 64, i * kBwdBlk, h0, b);
                    ptx::tma_load_4d(dst + 2 * kRowTile + dh * kRowTile, &tmG, bar(KV_QG_FULL + st), dh * 64, i * kBwdBlk, h0, b);
                }
                if (++hp == a.npairs) hp = 0;
            }
        }
        __syncwarp();
    } else if (warp == 1 || warp == 2) {
        // -------------------------------------------------------------- tcgen05 issuers of S (warp 1) and dP (warp 2)
        const bool leader = ptx::elect_one();
        const bool is_dp = __shfl_sync(0xffffffffu, warp, 0) == 2;
        constexpr uint32_t idesc_s = idesc_bf16(128, 64, 0, 0);    // both operands K-major
        // A = Q (S) or dO (dP) of the stage; B = the key block's K or V.
        const uint32_t b_lo = ((smem_base + (is_dp ? SM::kV : SM::kK)) >> 4) | (1u << 16);
        bool ok = __all_sync(0xffffffffu, wait_bar(bar(KV_KV_FULL), 0, 1));
        for (int e = 0; e < n && ok; ++e) {
            const uint32_t bf = e & 1;
            ok = __all_sync(0xffffffffu, wait_bar(bar(KV_QG_FULL + bf), (e >> 1) & 1, 3));
            if (ok && e >= 2) ok = __all_sync(0xffffffffu, wait_bar(bar(KV_S_TAKEN + bf), ((e >> 1) - 1) & 1, 4));
            if (!ok) break;
            ptx::tc_fence_after_sync();
            if (leader) {
                const uint32_t a_lo = ((smem_base + SM::kQG + bf * SM::kStage + (is_dp ? 2 * kRowTile : 0u)) >> 4) | (1u << 16);
                const uint32_t t_d = tmem_base + 128 * bf + (is_dp ? 64u : 0u);
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk)
                    ptx::umma_ss_lohi(t_d, a_lo + (((kk / 4) * kRowTile + (kk % 4) * 32) >> 4), kDescHi,
                                      b_lo + (((kk / 4) * kKeyTile + (kk % 4) * 32) >> 4), kDescHi, idesc_s, kk > 0 ? 1u : 0u);
                ptx::umma_commit(bar(KV_SD_FULL + bf));
            }
            __syncwarp();
        }
    } else if (warp == 3) {
        // -------------------------------------------------------------- tcgen05 issuer of dV^T and dK^T
        // (its own warp: a Q / dO stage is free for the next load only when these have read it, and a
        // single in-order issuer put them behind the next step's S and dP)
        const bool leader = ptx::elect_one();
        constexpr uint32_t idesc_t = idesc_bf16(128, 64, 1, 1);    // A feature-contiguous, B key-contiguous
        bool ok = true;
        for (int e1 = 0; e1 < n && ok; ++e1) {
            {
                const uint32_t bf = e1 & 1;
                ok = __all_sync(0xffffffffu, wait_bar(bar(KV_PD_FULL + bf), (e1 >> 1) & 1, 5));
                if (!ok) break;
                ptx::tc_fence_after_sync();
                if (leader) {
                    // A = the dO (Q) tile read feature-contiguous (its two 64-feature halves are kRowTile
                    // apart), B = P (dS) read key-contiguous; 16 tile rows per MMA, 2048 bytes further each.
                    const uint32_t qa = ((smem_base + SM::kQG + bf * SM::kStage) >> 4) | ((kRowTile >> 4) << 16);
                    const uint32_t ga = qa + ((2 * kRowTile) >> 4);
                    const uint32_t pb = ((smem_base + SM::kPD + bf * SM::kBuf) >> 4) | ((kRowTile >> 4) << 16);
                    const uint32_t db = pb + (kRowTile >> 4);
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)
                        ptx::umma_ss_lohi(tmem_base + kColDv, ga + ((kk * 2048) >> 4), kDescHi, pb + ((kk * 2048) >> 4), kDescHi,
                                          idesc_t, (e1 > 0 || kk > 0) ? 1u : 0u);
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)
                        ptx::umma_ss_lohi(tmem_base + kColDk, qa + ((kk * 2048) >> 4), kDescHi, db + ((kk * 2048) >> 4), kDescHi,
                                          idesc_t, (e1 > 0 || kk > 0) ? 1u : 0u);
                    ptx::umma_commit(bar(KV_QG_EMPTY + bf));  // (frees the P / dS buffer as well)
                    if (e1 == n - 1) ptx::umma_commit(bar(KV_DONE));
                }
                __syncwarp();
            }
        }
    } else if (warp >= 4) {
        // -------------------------------------------------------------- compute groups
        ptx::setmaxnreg_inc<PA_BWD_REG_COMP>();
        const int wg = (warp - 4) >> 2, quad = warp & 3;
        const int row = quad * 32 + lane, qrow = row & 63;
        const uint32_t t_lane = tmem_base + ((uint32_t)(quad * 32) << 16);
        // Row statistics of a step for this thread's row: LSE and delta; +inf / 0 for a row without
        // weights (beyond the sequence, padding head, empty row): P = 0.  Nothing here uses a loaded
        // value (the thread would wait for it on the spot): the query block index is loaded two of
        // this group's steps ahead, LSE and delta one step ahead, and they are looked at when the step
        // they belong to begins.
        auto step_block = [&](int e) { return e < n ? __ldg(a.row_idx + e0 + e / a.npairs) : -1; };
        auto request_stats = [&](int e, int32_t i, float &lse, float &delta, bool &diag) {
            lse = INFINITY;
            delta = 0.f;
            diag = false;
            if (e >= n) return;
            const int head_local = 2 * (e % a.npairs) + (row >> 6);
            const int64_t q = (int64_t)i * kBwdBlk + qrow;
            diag = i == j;
            if (head_local < a.G && q < a.N) {
                const int64_t at = ((int64_t)b * a.Hq + hk * a.G + head_local) * a.N + q;
                lse = __ldg(a.lse + at);
                delta = __ldg(a.delta + at);
            }
        };
        float lse_raw, delta, lse_raw_n, delta_n;
        bool diag, diag_n;
        int32_t i_next = step_block(wg + 2);
        request_stats(wg, step_block(wg), lse_raw, delta, diag);
        const uint32_t p_row = smem_base + SM::kPD + wg * SM::kBuf + (uint32_t)row * 128u;
        bool ok = true;
        for (int e = wg; e < n; e += 2) {
            const int32_t i_next2 = step_block(e + 4);
            request_stats(e + 2, i_next, lse_raw_n, delta_n, diag_n);  // (in flight during this step)
            ok = __all_sync(0xffffffffu, wait_bar(bar(KV_SD_FULL + wg), (e >> 1) & 1, 6));
            if (!ok) break;
            ptx::tc_fence_after_sync();
            uint32_t s[64], dp[64];
            ptx::tmem_ld32(t_lane + 128 * wg, *reinterpret_cast<uint32_t(*)[32]>(&s[0]));
            ptx::tmem_ld32(t_lane + 128 * wg + 32, *reinterpret_cast<uint32_t(*)[32]>(&s[32]));
            ptx::tmem_ld32(t_lane + 128 * wg + 64, *reinterpret_cast<uint32_t(*)[32]>(&dp[0]));
            ptx::tmem_ld32(t_lane + 128 * wg + 96, *reinterpret_cast<uint32_t(*)[32]>(&dp[32]));
            ptx::tmem_wait_ld();
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar(KV_S_TAKEN + wg));
            // (The P / dS buffer is free: the second products of step e - 2 that read it had completed
            // before this step's Q and dO could be loaded into the stage they also read, and so before
            // the S and dP waited for above were issued.)
            // Algorithm 1's causal term acts inside the diagonal pair only.
            const int lim = diag ? qrow : 63;
            const float lse2 = (lse_raw == -INFINITY || lse_raw == INFINITY) ? INFINITY : lse_raw * 1.4426950408889634f;
#pragma unroll
            for (int ch = 0; ch < 8; ++ch) {
                uint32_t pp[4], pd[4];
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    float p[2], ds[2];
#pragma unroll
                    for (int y = 0; y < 2; ++y) {
                        const int col = 8 * ch + 2 * x + y;
                        p[y] = (col <= lim) ? ptx::ex2(fmaf(__uint_as_float(s[col]), a.scale_log2, -lse2)) : 0.f;
                        ds[y] = p[y] * (__uint_as_float(dp[col]) - delta);
                    }
                    pp[x] = ptx::cvt_bf16x2(p[0], p[1]);
                    pd[x] = ptx::cvt_bf16x2(ds[0], ds[1]);
                }
                // 16-byte chunk ch of tile row r sits at chunk position ch ^ (r & 7) (128-byte swizzle).
                const uint32_t off = (uint32_t)((ch ^ (row & 7)) << 4);
                ptx::st_shared_v4(p_row + off, pp[0], pp[1], pp[2], pp[3]);
                ptx::st_shared_v4(p_row + kRowTile + off, pd[0], pd[1], pd[2], pd[3]);
            }
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar(KV_PD_FULL + wg));
            lse_raw = lse_raw_n;
            delta = delta_n;
            diag = diag_n;
            i_next = i_next2;
        }
        // Group 0 adds dK^T (x scale), group 1 dV^T: thread = feature, one key per register.
        if (ok) ok = __all_sync(0xffffffffu, wait_bar(bar(KV_DONE), 0, 8));
        if (ok) {
            ptx::tc_fence_after_sync();
            float *dst = (wg == 0 ? a.dk : a.dv) + (((int64_t)b * a.N + (int64_t)j * kBwdBlk) * a.Hkv + hk) * D + row;
            const float f = wg == 0 ? a.scale : 1.0f;
#pragma unroll
            for (int ch = 0; ch < 2; ++ch) {
                uint32_t acc[32];
                ptx::tmem_ld32(t_lane + (wg == 0 ? kColDk : kColDv) + 32 * ch, acc);
                ptx::tmem_wait_ld();
#pragma unroll
                for (int x = 0; x < 32; ++x) {
                    const int key = 32 * ch + x;
                    if ((int64_t)j * kBwdBlk + key < a.N) atomicAdd(dst + (int64_t)key * a.Hkv * D, __uint_as_float(acc[x]) * f);
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

// ---------------------------------------------------------------------------------- host side
template <int D>
static pa_status launch_dq(const BackwardArgs &a, const pa_prefill_params *p, const CUtensorMap &tmQ, const CUtensorMap &tmG,
                           const CUtensorMap &tmK, const CUtensorMap &tmV, int device, int sms, cudaStream_t st)
{
    CUtensorMap tmDq;
    const TensorMapKey out = {a.dq, p->seq_len, (int64_t)a.Hq * D, D, (int64_t)a.N * a.Hq * D, device, D, a.Hq, p->batch, 1, 32, 1};
    if (pa_status s = get_tensor_map(out, "dq", &tmDq)) return s;
    const int64_t n_items = (int64_t)a.nqb * a.Hkv * a.npairs * a.batch;
    if (n_items > (int64_t)0x3fffffff) return fail(PA_ERR_SHAPE, "too many work items (%lld)", (long long)n_items);
    dq_kernel<D><<<(unsigned)(n_items < sms ? n_items : sms), kDqThreads, DqCfg<D>::kAlloc, st>>>(tmQ, tmG, tmK, tmV, tmDq, a,
                                                                                                  (uint32_t)n_items);
    PA_CUDA_OK(cudaGetLastError());
    return PA_OK;
}

template <int D>
static pa_status launch_tc(const BackwardArgs &a, const pa_prefill_params *p, int64_t nnz, int device, int sms, cudaStream_t st)
{
    // Tensor maps (cached per buffer and shape): a Q or dO box holds the two heads of a tile, a K or V box one head.
    CUtensorMap tmQ, tmG, tmK, tmV;
    auto map_of = [&](const void *base, int heads, const pa_strides &s, int box_heads, const char *what, CUtensorMap *m) {
        const TensorMapKey key = {base, p->seq_len, s.seq, s.head, s.batch, device, D, heads, p->batch, box_heads, kBwdBlk, 0};
        return get_tensor_map(key, what, m);
    };
    if (pa_status s = map_of(a.q, a.Hq, p->q, 2, "q", &tmQ)) return s;
    if (pa_status s = map_of(a.d_o, a.Hq, p->o, 2, "d_o", &tmG)) return s;
    if (pa_status s = map_of(a.k, a.Hkv, p->k, 1, "k", &tmK)) return s;
    if (pa_status s = map_of(a.v, a.Hkv, p->v, 1, "v", &tmV)) return s;
    if (device_once_begin(device, D == 128 ? ONCE_BACKWARD_TC_ATTR : ONCE_BACKWARD_TC_ATTR_64)) {
        const cudaError_t e1 = cudaFuncSetAttribute(dq_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DqCfg<D>::kAlloc);
        const cudaError_t e2 = cudaFuncSetAttribute(dkv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DkvSmem::kAlloc);
        if (e1 != cudaSuccess || e2 != cudaSuccess) {
            device_once_reset(device, D == 128 ? ONCE_BACKWARD_TC_ATTR : ONCE_BACKWARD_TC_ATTR_64);
            return fail(PA_ERR_CUDA, "cudaFuncSetAttribute failed: %s", cudaGetErrorString(e1 != cudaSuccess ? e1 : e2));
        }
    }
    if (pa_status s = launch_dq<D>(a, p, tmQ, tmG, tmK, tmV, device, sms, st)) return s;
    if (D == 128) {
        // (an upper bound on the number of chunks; CTAs beyond the real count return at once)
        const int64_t max_chunks = nnz / a.chunk + a.nqb;
        dkv_kernel<<<dim3((unsigned)max_chunks, (unsigned)a.Hkv, (unsigned)a.batch), kTcThreads, DkvSmem::kAlloc, st>>>(tmQ, tmG, tmK, tmV, a);
        PA_CUDA_OK(cudaGetLastError());
    }
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
