// Query-major passes of the backward (paper Section 4.2, "The Backward Pass": one kernel reduces dQ over keys, the
// other reduces dK and dV over queries; the probability matrix is rebuilt from the saved log-sum-exp, never stored):
//   attn_dq_kernel     dQ_i = scale * sum_j dS_ij K_j,  dS = exp2(S*c - LSE*log2e) * (dP - Delta).  Every dQ row is
//                      summed by one thread block in key order: no atomics, no workspace, bitwise reproducible.
//   attn_delta_kernel  Delta_i = sum_j P_ij (dO_i . V_j): the exact softmax-Jacobian row term.  The cheap route to the
//                      same quantity, rowsum(dO * O), inherits the bf16 rounding of the stored O, which with sharply
//                      peaked rows (|O| ~ |V|) is the largest term in dQ and dK.
// dQ at D=128 only, the exact Delta there and, in the smallest and the largest problems, at D=64 (elsewhere: attn_dq64.cu).
// Both form S = Q K_j^T and dP = dO V_j^T tile by tile and differ in what becomes of the tile, so they are two builds of
// one kernel.
//
// A work item is a block of 256 query rows of one head: two 128-row tiles, A and B, that share every K and V tile
// they both need; in small problems one tile (plan_of).  The keys go by in steps of 64.  Items are handed out dynamically,
// heaviest first, as in the forward (WorkRing).  384 threads:
//   warp 0      TMA producer: Q and dO per tile of an item, K and V through a ring of 64-key stages
//   warps 1, 3  UMMA issuers, one per query tile, so that neither tile waits for the other's products and A may be in
//               the next item while B finishes this one
//   warps 4-7   rows of tile A, warps 8-11 rows of tile B: one thread per query row takes 64 keys of S and dP out of
//               tensor memory and writes dS back as bf16 (or adds P*dP into its Delta)
// (with single tiles, tile B's warps have nothing to do)
//
// What bounds it: one tile in flight is a serial chain (products -> tensor memory -> arithmetic -> tensor memory ->
// product), during which the tensor cores idle; two tiles fill each other's gaps.  64 keys per step is what tensor memory
// allows two tiles at D=128: dQ takes 128 of a tile's 256 columns, S and dP 64 each.  A product of N=64 with both
// operands in shared memory costs 49 clocks per 16 k elements against 65 for twice the keys, so a 128 x 128 block takes
// 2100 clocks of tensor time at D=128 (1560 with N=128).
#include <algorithm>
#include <type_traits>

#include "kernels.h"
#include "ptx.cuh"

namespace nova {
namespace {

constexpr int kThreads = 384;
constexpr int kTmemCols = 512;
constexpr int kStep = kKeyStep;                  // keys per step
constexpr int kHalfStepBytes = kStep * 128;      // one [64 keys x 64 bf16] box

// kTiles: query tiles of a work item (see plan_of).
template <int D, int kTiles>
struct DqCfg {
    static constexpr int kBlockRows = kTiles * kBlockQ;   // query rows per work item
    static constexpr int kWorkConsumers = kTiles * 5;     // an issuer and four row warps per tile
    static constexpr int kHalves = D / kBoxCols;
    static constexpr int kTileBytes = kHalves * kHalfTileBytes;
    static constexpr int kStepBytes = kHalves * kHalfStepBytes;
    static constexpr int kQStages = (D == 64 || kTiles == 1) ? 2 : 1;  // Q and dO of an item
    static constexpr int kKVStages = (D == 64) ? 5 : 3;
    static constexpr int kOffQ = 0;                                     // [kQStages][kTiles] of Q, then of dO
    static constexpr int kOffdO = kQStages * kTiles * kTileBytes;
    static constexpr int kOffK = 2 * kOffdO;                            // [kKVStages] of K, then of V
    static constexpr int kOffV = kOffK + kKVStages * kStepBytes;
    static constexpr int kOffBar = kOffV + kKVStages * kStepBytes;
    static constexpr int kSmemBytes = kOffBar + 512 + 1024;
    static_assert(kSmemBytes <= 232448, "exceeds the shared memory of one CTA");
    // Columns of a tile (256 per tile of a pair).  dQ first, then S and dP.  Where there is room two buffers of dS (32
    // columns each), so that S and dP of the next step are queued as soon as the row warps have read them; with two tiles
    // dS lies over S.
    static constexpr bool kSepdS = kTiles == 1;
    static constexpr int kColS = D, kColdP = D + 64;
    static constexpr int kColdS = kSepdS ? D + 128 : kColS;
};

struct DqBars {
    uint64_t q_full[2][2], q_empty[2][2];  // [stage][tile]
    uint64_t kv_full[5], kv_empty[5];
    uint64_t sp_full[2][2], sp_free[2][2];  // [buffer][tile]; the second buffer is used by the Delta build only
    // Two ds_ready per tile, used in turn: where dS has columns of its own the row warps may finish step j + 1 before the
    // issuer has seen step j, and a single barrier two phases on looks as if it had not moved.
    uint64_t ds_ready[2][2];                     // [step & 1][tile]
    uint64_t dq_done[2], dq_free[2], staged[2];  // per tile
    uint64_t drain[2];
    WorkRing ring;
    uint32_t tmem_base;
    int abort_flag;
};
static_assert(sizeof(DqBars) <= 512, "barrier block");

// Work items: blocks of kTiles query tiles, heaviest first (the last block of a causal problem sees every key).  D=128: within
// chunks of heads whose tensors stay in L2 together (the exact Delta at B=16, H=32, T=1024 175 -> 157 us, the
// deterministic backward 650 -> 627 us); at D=64 a head's K and V are half as large and the longer arithmetic costs
// 1 % where there is nothing to gain.
template <int D, int kTiles>
struct DqWork {
    int BH, n_blocks, chunk, T, H;
    uint32_t orders;  // coordinate orders of the Q, K, V, dO, dQ tensor maps, four bits each
    bool causal;
    // Block index, head, and the number of key steps each tile visits (0: the tile lies past the end of the sequence).
    __device__ __forceinline__ void get(int idx, int* blk, int* bh, int* n_a, int* n_b) const {
        if constexpr (D == 128) {
            int first = 0, in = idx, heads = BH;  // first head of the chunk, item within it, its heads
            if (chunk < BH) {
                const int per_chunk = chunk * n_blocks, ck = idx / per_chunk;
                first = ck * chunk;
                in = idx - ck * per_chunk;
                heads = min(chunk, BH - first);
            }
            const int order = in / heads;
            *blk = n_blocks - 1 - order;
            *bh = first + in - order * heads;
        } else {
            *blk = n_blocks - 1 - idx / BH;
            *bh = idx % BH;
        }
        const int n_all = (T + kStep - 1) / kStep;
        const int qt_a = kTiles * (*blk), qt_b = qt_a + 1;
        *n_a = causal ? min((qt_a + 1) * (kBlockQ / kStep), n_all) : n_all;
        *n_b = (kTiles == 2 && qt_b * kBlockQ < T) ? (causal ? min((qt_b + 1) * (kBlockQ / kStep), n_all) : n_all) : 0;
    }
};

template <int D, int kTiles, bool kStrided>
__device__ __forceinline__ void dq_producer(const CUtensorMap* tmQ, const CUtensorMap* tmK, const CUtensorMap* tmV,
                                            const CUtensorMap* tmdO, uint8_t* smem, DqBars* bars, const DqWork<D, kTiles>& wk) {
    using Cfg = DqCfg<D, kTiles>;
    volatile int* abort_flag = &bars->abort_flag;
    constexpr long long limit = kWaitLimitCycles;
    int armed_q[2][2] = {{-1, -1}, {-1, -1}}, armed_kv[Cfg::kKVStages];
    for (int s = 0; s < Cfg::kKVStages; ++s) armed_kv[s] = -1;
    bool ok = true, clc_pending = false;
    int w = 0, st = 0;  // items so far, K/V stage
    uint32_t ph = 0;    // and its phase
    int item = blockIdx.x;
    for (;;) {
        ok = bars->ring.publish(w, item, abort_flag, limit);
        if (!ok || item < 0) break;
        int blk, bh, n_a, n_b;
        wk.get(item, &blk, &bh, &n_a, &n_b);
        const int head = kStrided ? bh % wk.H : 0, batch = kStrided ? bh / wk.H : 0;
        const int qs = w % Cfg::kQStages;
        const uint32_t qph = (w / Cfg::kQStages) & 1;
        const int n = max(n_a, n_b);
        // Tile A's Q and dO, the first keys, tile B's Q and dO (whose buffers tile B hands back later than A), the rest.
        auto load_q = [&](int t) -> bool {
            if (!mbar_wait(&bars->q_empty[qs][t], qph ^ 1, abort_flag)) return false;
            mbar_expect_tx(&bars->q_full[qs][t], 2 * Cfg::kTileBytes);  // rows past T arrive as zeros
            armed_q[qs][t] = qph;
#pragma unroll
            for (int h = 0; h < Cfg::kHalves; ++h) {
                const int off = (qs * kTiles + t) * Cfg::kTileBytes + h * kHalfTileBytes;
                tma_load_tile<kStrided>(smem + Cfg::kOffQ + off, tmQ, &bars->q_full[qs][t], wk.orders & 15, h * kBoxCols,
                                        blk * Cfg::kBlockRows + t * kBlockQ, head, batch, bh);
                tma_load_tile<kStrided>(smem + Cfg::kOffdO + off, tmdO, &bars->q_full[qs][t], (wk.orders >> 12) & 15,
                                        h * kBoxCols, blk * Cfg::kBlockRows + t * kBlockQ, head, batch, bh);
            }
            return true;
        };
        ok = load_q(0);
        if (!ok) break;
        for (int j = 0; j < n; ++j) {
            ok = mbar_wait(&bars->kv_empty[st], ph ^ 1, abort_flag);
            if (!ok) break;
            mbar_expect_tx(&bars->kv_full[st], 2 * Cfg::kStepBytes);
            armed_kv[st] = ph;
#pragma unroll
            for (int h = 0; h < Cfg::kHalves; ++h) {
                tma_load_tile<kStrided>(smem + Cfg::kOffK + st * Cfg::kStepBytes + h * kHalfStepBytes, tmK,
                                        &bars->kv_full[st], (wk.orders >> 4) & 15, h * kBoxCols, j * kStep, head, batch, bh);
                tma_load_tile<kStrided>(smem + Cfg::kOffV + st * Cfg::kStepBytes + h * kHalfStepBytes, tmV,
                                        &bars->kv_full[st], (wk.orders >> 8) & 15, h * kBoxCols, j * kStep, head, batch, bh);
            }
            if (++st == Cfg::kKVStages) {
                st = 0;
                ph ^= 1;
            }
            if (kTiles == 2 && j == 0) {
                ok = load_q(1);
                if (!ok) break;
            }
        }
        if (!ok) break;
        // all loads of this item are on their way: claim the next one now, and no earlier
        bars->ring.request();
        clc_pending = true;
        ok = bars->ring.answer(w, &item, abort_flag, limit);
        if (!ok) break;
        clc_pending = false;
        ++w;
    }
    if (!ok) {  // giving up: let what is in flight land before the CTA's shared memory goes away
        int none = 0;
        if (clc_pending) (void)mbar_wait(&bars->ring.answer_bar, w & 1, &none);
        for (int s = 0; s < 2; ++s)
            for (int t = 0; t < kTiles; ++t)
                if (armed_q[s][t] >= 0) (void)mbar_wait(&bars->q_full[s][t], armed_q[s][t], &none);
        for (int s = 0; s < Cfg::kKVStages; ++s)
            if (armed_kv[s] >= 0) (void)mbar_wait(&bars->kv_full[s], armed_kv[s], &none);
    }
}

// The issuer of query tile t: the whole warp in uniform control flow, one elected lane issues.
template <int D, int kTiles, bool kDelta>
__device__ __forceinline__ void dq_mma(uint8_t* smem, DqBars* bars, uint32_t tmem_base, const DqWork<D, kTiles>& wk, int t) {
    using Cfg = DqCfg<D, kTiles>;
    volatile int* abort_flag = &bars->abort_flag;
    constexpr uint32_t kIdescT = umma_idesc_bf16(128, kStep, 0, 0);  // S, dP
    constexpr uint32_t kIdescdQ = umma_idesc_bf16(128, D, 0, 1);     // dQ: A from TMEM, B (K) MN-major
    const uint32_t hi = umma_desc_hi_sw128(1024);
    const uint32_t k_k0 = umma_desc_lo(smem_u32(smem + Cfg::kOffK), 16);
    const uint32_t v_k0 = umma_desc_lo(smem_u32(smem + Cfg::kOffV), 16);
    const uint32_t k_m0 = umma_desc_lo(smem_u32(smem + Cfg::kOffK), kHalfStepBytes);
    const uint32_t t_dq = tmem_base + 256 * t;
    const bool el = elect_one();
    const int lane = threadIdx.x & 31;
    bool ok = true;
    int w = 0, wt = 0;  // items; items in which the tile took part
    int c = 0, cq = 0;  // steps of this tile finished; steps whose S and dP have been issued
    int st = 0;         // K/V stage of the current step
    uint32_t ph = 0;    // and its phase
    uint32_t q_k = 0, do_k = 0;

    // acc[64 columns] = A_t B^T with both operands K-major, 16 head-dim elements (32 bytes) per instruction
    auto product = [&](uint32_t t_acc, uint32_t a, uint32_t b) {
#pragma unroll
        for (int k = 0; k < D / 16; ++k)
            umma_ss(t_acc, umma_desc_join(a + (((k / 4) * kHalfTileBytes + (k % 4) * 32) >> 4), hi),
                    umma_desc_join(b + (((k / 4) * kHalfStepBytes + (k % 4) * 32) >> 4), hi), kIdescT, k > 0 ? 1u : 0u);
    };
    auto next_stage = [&](int* s, uint32_t* p) {
        if (++*s == Cfg::kKVStages) {
            *s = 0;
            *p ^= 1;
        }
    };

    for (;;) {
        const int item = bars->ring.take(w, lane, abort_flag, kWaitLimitCycles);
        if (item < 0) {
            ok = (item == -1);
            break;
        }
        int blk, bh, n_a, n_b;
        wk.get(item, &blk, &bh, &n_a, &n_b);
        const int n_t = t == 0 ? n_a : n_b, n = max(n_a, n_b);
        const int qs = w % Cfg::kQStages;
        q_k = umma_desc_lo(smem_u32(smem + Cfg::kOffQ + (qs * kTiles + t) * Cfg::kTileBytes), 16);
        do_k = umma_desc_lo(smem_u32(smem + Cfg::kOffdO + (qs * kTiles + t) * Cfg::kTileBytes), 16);
        if (n_t > 0) {
            ok = mbar_wait(&bars->q_full[qs][t], (w / Cfg::kQStages) & 1, abort_flag);
            if (!ok) break;
        }
        if constexpr (kDelta) {
            for (int j = 0; j < n_t; ++j, ++cq) {
                ok = mbar_wait(&bars->kv_full[st], ph, abort_flag);
                // the row warps have read what this buffer held two steps ago
                if (ok) ok = mbar_wait(&bars->sp_free[cq & 1][t], ((cq >> 1) & 1) ^ 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                if (el) {
                    const uint32_t t_s = tmem_base + 256 * t + 128 * (cq & 1);
                    product(t_s, q_k, k_k0 + st * (Cfg::kStepBytes >> 4));
                    product(t_s + 64, do_k, v_k0 + st * (Cfg::kStepBytes >> 4));
                    tc_commit(&bars->sp_full[cq & 1][t]);
                    tc_commit(&bars->kv_empty[st]);
                    if (j + 1 == n_t) tc_commit(&bars->q_empty[qs][t]);
                }
                __syncwarp();
                next_stage(&st, &ph);
            }
        } else {
            const uint32_t t_s = t_dq + Cfg::kColS, t_dp = t_dq + Cfg::kColdP;
            int st_n = st;  // stage of the step whose S and dP come next
            uint32_t ph_n = ph;
            // S and dP of the item's first step.  Their columns are free: the row warps have read the previous step's
            // (sp_free was awaited below, or is here), and a dS that lies over S was consumed by a dQ product queued
            // earlier.
            if (n_t > 0) {
                ok = mbar_wait(&bars->kv_full[st_n], ph_n, abort_flag);
                if (ok && cq > 0) ok = mbar_wait(&bars->sp_free[0][t], (cq - 1) & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                if (el) {
                    product(t_s, q_k, k_k0 + st_n * (Cfg::kStepBytes >> 4));
                    product(t_dp, do_k, v_k0 + st_n * (Cfg::kStepBytes >> 4));
                    tc_commit(&bars->sp_full[0][t]);
                }
                __syncwarp();
                ++cq;
                next_stage(&st_n, &ph_n);
            }
            for (int j = 0; j < n_t; ++j, ++c) {
                const bool more = j + 1 < n_t;
                if (more) {  // dP (and S, where dS has columns of its own) of the next step, once this step's have been read
                    ok = mbar_wait(&bars->kv_full[st_n], ph_n, abort_flag);
                    if (ok) ok = mbar_wait(&bars->sp_free[0][t], (cq - 1) & 1, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    if (el) {
                        if (Cfg::kSepdS) product(t_s, q_k, k_k0 + st_n * (Cfg::kStepBytes >> 4));
                        product(t_dp, do_k, v_k0 + st_n * (Cfg::kStepBytes >> 4));
                        if (Cfg::kSepdS) tc_commit(&bars->sp_full[0][t]);
                    }
                    __syncwarp();
                }
                ok = mbar_wait(&bars->ds_ready[c & 1][t], (c >> 1) & 1, abort_flag);
                // the previous item's dQ must have been read out of TMEM before it is overwritten
                if (ok && j == 0 && wt > 0) ok = mbar_wait(&bars->dq_free[t], (wt - 1) & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                // dQ += dS K_j: dS from TMEM (16 keys = 8 packed columns per instruction), K MN-major (rows = keys,
                // 64 head-dim elements per 128-byte row, the second 64-wide half kHalfStepBytes further).
                if (el) {
                    const uint32_t t_ds = t_dq + Cfg::kColdS + (Cfg::kSepdS ? 32 * (c & 1) : 0);
                    const uint32_t k_m = k_m0 + st * (Cfg::kStepBytes >> 4);
#pragma unroll
                    for (int k = 0; k < kStep / 16; ++k)
                        umma_ts(t_dq, t_ds + k * 8, umma_desc_join(k_m + k * 128, hi), kIdescdQ, (j > 0 || k > 0) ? 1u : 0u);
                    tc_commit(&bars->kv_empty[st]);
                    if (!more) tc_commit(&bars->dq_done[t]);
                    if (!Cfg::kSepdS && more) {  // S of the next step, over the dS that the product above reads
                        product(t_s, q_k, k_k0 + st_n * (Cfg::kStepBytes >> 4));
                        tc_commit(&bars->sp_full[0][t]);
                    }
                }
                __syncwarp();
                if (more) {
                    ++cq;
                    next_stage(&st_n, &ph_n);
                }
                next_stage(&st, &ph);
            }
        }
        if (!ok) break;
        // Steps that only the other tile visits: this tile's share of their release, each once it has landed (an earlier
        // arrival could fall into the stage's previous use).
        for (int j = n_t; j < n; ++j) {
            ok = mbar_wait(&bars->kv_full[st], ph, abort_flag);
            if (!ok) break;
            if (lane == 0) mbar_arrive(&bars->kv_empty[st]);
            __syncwarp();
            next_stage(&st, &ph);
        }
        if (!ok) break;
        if (n_t > 0) ++wt;
        ++w;
    }
    if (!ok) {
        int none = 0;
        if (el) tc_commit(&bars->drain[t]);
        __syncwarp();
        (void)mbar_wait(&bars->drain[t], 0, &none);
    }
}

// The row warps of query tile t.
template <int D, int kTiles, bool kCausal, bool kStrided, bool kDelta>
__device__ __forceinline__ void dq_rows(uint8_t* smem, DqBars* bars, uint32_t tmem_base, const CUtensorMap* tmdQ,
                                        const float* __restrict__ LSE, const float* __restrict__ Delta,
                                        float* __restrict__ Delta_out, float scale, const DqWork<D, kTiles>& wk, int t, int rwarp,
                                        int lane) {
    using Cfg = DqCfg<D, kTiles>;
    volatile int* abort_flag = &bars->abort_flag;
    const uint32_t lane_base = 32u * rwarp;
    const int row_local = lane_base + lane;
    const bool leader = (rwarp == 0 && lane == 0);
    const uint32_t t_dq = tmem_addr(tmem_base, lane_base, 256 * t);
    const float c = scale * kLog2e;
    const uint64_t c2 = f32x2_pack(c, c);
    const int T = wk.T;
    bool ok = true;
    int w = 0, wt = 0, cnt = 0;  // items, items this tile took part in, steps processed by this tile
    int pending_qs = -1;         // Q stage whose dQ store was issued at the end of the previous item

    for (;;) {
        const int item = bars->ring.take(w, lane, abort_flag, kWaitLimitCycles);
        if (item < 0) {
            ok = (item == -1);
            break;
        }
        int blk, bh, n_a, n_b;
        wk.get(item, &blk, &bh, &n_a, &n_b);
        const int n_t = (t == 0) ? n_a : n_b;
        const int qt = kTiles * blk + t;
        const int row = qt * kBlockQ + row_local;
        const size_t idx = static_cast<size_t>(bh) * T + row;
        const int qs = w % Cfg::kQStages;
        if (n_t == 0) {  // tile past the end of the sequence: only release its buffers, once they have been filled
            bool leader_ok = true;
            if (leader) {
                if (pending_qs >= 0) {
                    bulk_wait_group_read<0>();
                    mbar_arrive(&bars->q_empty[pending_qs][t]);
                }
                leader_ok = mbar_wait(&bars->q_full[qs][t], (w / Cfg::kQStages) & 1, abort_flag);
                if (leader_ok) mbar_arrive(&bars->q_empty[qs][t]);
            }
            pending_qs = -1;
            ok = __all_sync(0xffffffffu, leader_ok);
            if (!ok) break;
            ++w;
            continue;
        }
        // Rows past the end of the sequence: LSE = +inf gives P = 0 everywhere.
        const float nlse2 = (row < T) ? -LSE[idx] * kLog2e : -INFINITY;
        const float ndelta = (!kDelta && row < T) ? -Delta[idx] : 0.f;
        const uint64_t nlse = f32x2_pack(nlse2, nlse2), nd = f32x2_pack(ndelta, ndelta);
        uint64_t acc0 = 0, acc1 = 0;
        // D=64: steps in turn, as the two groups of the other kernel for this head dimension (attn_dq64.cu) sum them: which of the
        // two a call takes depends on the number of heads, the bits of a head do not.
        constexpr bool kInTurn = (D == 64);
        uint64_t next0 = 0, next1 = 0;

        for (int j = 0; j < n_t; ++j, ++cnt) {
            const int buf = kDelta ? (cnt & 1) : 0;
            ok = mbar_wait(&bars->sp_full[buf][t], (kDelta ? (cnt >> 1) : cnt) & 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            const uint32_t t_s = t_dq + (kDelta ? 128 * buf : Cfg::kColS);
            const uint32_t t_dp = kDelta ? t_s + 64 : t_dq + Cfg::kColdP;
            uint32_t sv[kStep], dv[kStep];
            tmem_ld_x32(t_s, sv);
            tmem_ld_x32(t_s + 32, sv + 32);
            tmem_ld_x32(t_dp, dv);
            tmem_ld_x32(t_dp + 32, dv + 32);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->sp_free[buf][t]);
            // Mask from indices only: causal keeps key <= query, the end of the sequence key < T.
            const int lim = (kCausal ? min(row, T - 1) : T - 1) - j * kStep;  // last kept key of the step
            if ((kCausal && (j + 1) * kStep > qt * kBlockQ) || (j + 1) * kStep > T) {
#pragma unroll
                for (int i = 0; i < kStep; ++i)
                    if (i > lim) sv[i] = 0xff800000u;  // -inf: P = 0
            }
            uint32_t ds[kStep / 2];
#pragma unroll
            for (int i = 0; i < kStep; i += 4) {
                float x0, x1, x2, x3;
                f32x2_unpack(f32x2_fma(f32x2_pack(__uint_as_float(sv[i + 0]), __uint_as_float(sv[i + 1])), c2, nlse), x0, x1);
                f32x2_unpack(f32x2_fma(f32x2_pack(__uint_as_float(sv[i + 2]), __uint_as_float(sv[i + 3])), c2, nlse), x2, x3);
                const uint64_t p01 = f32x2_pack(ex2_approx(x0), ex2_approx(x1)), p23 = f32x2_pack(ex2_approx(x2), ex2_approx(x3));
                const uint64_t d01 = f32x2_pack(__uint_as_float(dv[i + 0]), __uint_as_float(dv[i + 1]));
                const uint64_t d23 = f32x2_pack(__uint_as_float(dv[i + 2]), __uint_as_float(dv[i + 3]));
                if constexpr (kDelta) {
                    acc0 = f32x2_fma(p01, d01, acc0);
                    acc1 = f32x2_fma(p23, d23, acc1);
                } else {
                    f32x2_unpack(f32x2_mul(p01, f32x2_add(d01, nd)), x0, x1);
                    f32x2_unpack(f32x2_mul(p23, f32x2_add(d23, nd)), x2, x3);
                    ds[i / 2] = pack_bf16x2(x0, x1);
                    ds[i / 2 + 1] = pack_bf16x2(x2, x3);
                }
            }
            if constexpr (kDelta && kInTurn) {
                const uint64_t a0 = acc0, a1 = acc1;
                acc0 = next0, acc1 = next1;
                next0 = a0, next1 = a1;
            }
            if constexpr (!kDelta) {
                // Single tiles: the dQ product of two steps ago, which read this buffer, was queued before S of this step, and
                // the tensor pipe completes in order.
                tmem_st_x32(t_dq + Cfg::kColdS + (Cfg::kSepdS ? 32 * (cnt & 1) : 0), ds);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars->ds_ready[cnt & 1][t]);
                if (pending_qs >= 0) {
                    if (leader) {
                        bulk_wait_group_read<0>();
                        mbar_arrive(&bars->q_empty[pending_qs][t]);
                    }
                    pending_qs = -1;
                    __syncwarp();
                }
            }
        }
        if (!ok) break;
        if constexpr (kDelta) {
            float a0, a1, a2, a3;
            f32x2_unpack(acc0, a0, a1);
            f32x2_unpack(acc1, a2, a3);
            float sum = (a0 + a1) + (a2 + a3);
            if constexpr (kInTurn) {
                f32x2_unpack(next0, a0, a1);
                f32x2_unpack(next1, a2, a3);
                sum += (a0 + a1) + (a2 + a3);
            }
            if (row < T) Delta_out[idx] = sum;
            __syncwarp();
        } else {
            // ---- end of the item: scale * dQ_t as bf16 into this tile's Q buffer (no longer read: the last dQ product
            // completed after every S of the tile), then TMA stores
            ok = mbar_wait(&bars->dq_done[t], wt & 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            uint8_t* stage = smem + Cfg::kOffQ + (qs * kTiles + t) * Cfg::kTileBytes;
#pragma unroll
            for (int cb = 0; cb < D; cb += 32) {
                uint32_t a[32];
                tmem_ld_x32(t_dq + cb, a);
                tmem_wait_ld();
                uint8_t* row_ptr = stage + (cb / 64) * kHalfTileBytes + row_local * 128;
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const int ch = (cb % 64) / 8 + x;  // 16-byte chunk of the 128-byte swizzled row
                    uint4 v;
                    v.x = pack_bf16x2(__uint_as_float(a[8 * x + 0]) * scale, __uint_as_float(a[8 * x + 1]) * scale);
                    v.y = pack_bf16x2(__uint_as_float(a[8 * x + 2]) * scale, __uint_as_float(a[8 * x + 3]) * scale);
                    v.z = pack_bf16x2(__uint_as_float(a[8 * x + 4]) * scale, __uint_as_float(a[8 * x + 5]) * scale);
                    v.w = pack_bf16x2(__uint_as_float(a[8 * x + 6]) * scale, __uint_as_float(a[8 * x + 7]) * scale);
                    *reinterpret_cast<uint4*>(row_ptr + ((ch ^ (row_local & 7)) << 4)) = v;
                }
            }
            tc_fence_before();
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&bars->dq_free[t]);
                mbar_arrive(&bars->staged[t]);
            }
            bool leader_ok = true;
            if (leader) {
                leader_ok = mbar_wait(&bars->staged[t], wt & 1, abort_flag);
                if (leader_ok) {
#pragma unroll
                    for (int h = 0; h < Cfg::kHalves; ++h)
                        tma_store_tile<kStrided>(tmdQ, stage + h * kHalfTileBytes, (wk.orders >> 16) & 15, h * kBoxCols,
                                                 qt * kBlockQ, kStrided ? bh % wk.H : 0, kStrided ? bh / wk.H : 0, bh);
                    bulk_commit_group();
                    if (Cfg::kQStages == 1) {  // the next item's Q tile needs this very buffer
                        bulk_wait_group_read<0>();
                        mbar_arrive(&bars->q_empty[qs][t]);
                    }
                }
            }
            if (Cfg::kQStages > 1) pending_qs = qs;  // handed back after the next item's first step, as in the forward
            ok = __all_sync(0xffffffffu, leader_ok);
            if (!ok) break;
        }
        ++w;
        ++wt;
    }
    if (!kDelta && leader) bulk_wait_group<0>();  // dQ must be complete before the kernel ends
}

// Set-up and roles, shared by the two builds below.
template <int D, int kTiles, bool kCausal, bool kStrided, bool kDelta>
__device__ __forceinline__ void dq_body(const CUtensorMap* tmQ, const CUtensorMap* tmK, const CUtensorMap* tmV,
                                        const CUtensorMap* tmdO, const CUtensorMap* tmdQ, const float* __restrict__ LSE,
                                        const float* __restrict__ Delta, float* __restrict__ Delta_out, const DqWork<D, kTiles>& wk,
                                        float scale, int* __restrict__ dev_status) {
    using Cfg = DqCfg<D, kTiles>;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    DqBars* bars = reinterpret_cast<DqBars*>(smem + Cfg::kOffBar);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int t = 0; t < 2; ++t) {
            for (int s = 0; s < 2; ++s) {
                mbar_init(&bars->q_full[s][t], 1);
                mbar_init(&bars->q_empty[s][t], 1);
                mbar_init(&bars->sp_full[s][t], 1);
                mbar_init(&bars->sp_free[s][t], 4);
                mbar_init(&bars->ds_ready[s][t], 4);
            }
            mbar_init(&bars->dq_done[t], 1);
            mbar_init(&bars->dq_free[t], 4);
            mbar_init(&bars->staged[t], 4);
            mbar_init(&bars->drain[t], 1);
        }
        for (int s = 0; s < Cfg::kKVStages; ++s) {
            mbar_init(&bars->kv_full[s], 1);
            mbar_init(&bars->kv_empty[s], kTiles);  // the issuers
        }
        bars->ring.init(Cfg::kWorkConsumers);
        bars->abort_flag = 0;
        fence_mbar_init();
        tma_prefetch_desc(tmQ);
        tma_prefetch_desc(tmK);
        tma_prefetch_desc(tmV);
        tma_prefetch_desc(tmdO);
        if (!kDelta) tma_prefetch_desc(tmdQ);
    }
    if (warp == 1) {
        tmem_alloc(&bars->tmem_base, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = bars->tmem_base;
    griddep_launch_dependents();
    griddep_wait();  // everything above overlaps the previous kernel of the stream

    if (warp == 0) {
        if (lane == 0) dq_producer<D, kTiles, kStrided>(tmQ, tmK, tmV, tmdO, smem, bars, wk);
    } else if (warp == 1 || (kTiles == 2 && warp == 3)) {
        dq_mma<D, kTiles, kDelta>(smem, bars, tmem_base, wk, warp >> 1);
    } else if (warp >= 4 && warp < 4 + 4 * kTiles) {
        dq_rows<D, kTiles, kCausal, kStrided, kDelta>(smem, bars, tmem_base, tmdQ, LSE, Delta, Delta_out, scale, wk,
                                                      (warp - 4) >> 2, warp & 3, lane);
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, kTmemCols);
    if (threadIdx.x == 0 && bars->abort_flag != 0) atomicExch(dev_status, kDevTimeout);
}

template <int D, int kTiles, bool kCausal, bool kStrided>
__global__ void __launch_bounds__(kThreads, 1)
attn_dq_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
               const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmdO,
               const __grid_constant__ CUtensorMap tmdQ, const float* __restrict__ LSE, const float* __restrict__ Delta,
               int T, int BH, int H, uint32_t orders, int n_blocks, int chunk, float scale, int* __restrict__ dev_status) {
    dq_body<D, kTiles, kCausal, kStrided, false>(&tmQ, &tmK, &tmV, &tmdO, &tmdQ, LSE, Delta, nullptr,
                                                 DqWork<D, kTiles>{BH, n_blocks, chunk, T, H, orders, kCausal}, scale, dev_status);
}

template <int D, int kTiles, bool kCausal>
__global__ void __launch_bounds__(kThreads, 1)
attn_delta_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                  const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmdO,
                  const float* __restrict__ LSE, float* __restrict__ Delta, int T, int BH, int n_blocks, int chunk, float scale,
                  int* __restrict__ dev_status) {
    dq_body<D, kTiles, kCausal, false, true>(&tmQ, &tmK, &tmV, &tmdO, nullptr, LSE, nullptr, Delta,
                                             DqWork<D, kTiles>{BH, n_blocks, chunk, T, 1, 0u, kCausal}, scale, dev_status);
}

// Key steps after which the last SM is done.  Every item costs two besides its own.
long long span_of(const AttnShape& s, int tiles, int n_blocks, int num_sms) {
    const long long BH = static_cast<long long>(s.B) * s.H, n_all = (s.T + kStep - 1) / kStep;
    return steps_until_done(n_blocks * BH, num_sms, [&](long long idx) {
        const long long blk = n_blocks - 1 - idx / BH;
        return 2 + (s.causal ? std::min(tiles * (blk + 1) * (kBlockQ / kStep), n_all) : n_all);
    });
}

// How many tiles an item has, and what follows from it.
//
// Two tiles share their K and V and fill each other's gaps, which is worth 30 to 40 % of the work where there is enough of
// it; a tile alone takes a step in 0.6 of a pair's time, so it wins where the longest chain or the last round of items
// decides.  The weights 5:8 are fitted to both forms' times over 688 shapes (T = 129 to 8192, 40 to 1200 tiles, with and
// without the mask, both head dimensions): the slower form is taken at a mean cost of 0.3 %.  Pairs against single tiles,
// exact Delta: H=8, T=4096: 69.4, 41.8 us.  (What comes here at D=64 is either one tile a head or many pairs.)
struct Plan {
    int tiles, n_blocks, chunk;
    dim3 grid;  // one CTA per item; those that do not start at once are taken over by those that did
};
Plan plan_of(const AttnShape& s, int num_sms) {
    Plan p;
    const int n_tiles = (s.T + kBlockQ - 1) / kBlockQ, n_pairs = (n_tiles + 1) / 2, BH = s.B * s.H;
    p.tiles = 2;
    if (static_cast<long long>(n_pairs) * BH <= 4ll * num_sms) {  // (beyond that pairs always win, and the sum stays short)
        const long long one = span_of(s, 1, n_tiles, num_sms), two = span_of(s, 2, n_pairs, num_sms);
        if (5 * one < 8 * two) p.tiles = 1;
    }
    p.n_blocks = (n_tiles + p.tiles - 1) / p.tiles;
    p.chunk = heads_per_chunk(BH, p.n_blocks, s.T, s.D, num_sms);
    p.grid = dim3(static_cast<unsigned>(p.n_blocks) * BH);
    return p;
}

// Calls f with the head dimension, the tiles of an item and the mask as compile-time constants.
template <typename F>
cudaError_t dispatch(int D, int tiles, bool causal, F&& f) {
    auto with_d = [&](auto d) {
        auto with_tiles = [&](auto t) { return causal ? f(d, t, std::true_type{}) : f(d, t, std::false_type{}); };
        return tiles == 1 ? with_tiles(std::integral_constant<int, 1>{}) : with_tiles(std::integral_constant<int, 2>{});
    };
    return D == 64 ? with_d(std::integral_constant<int, 64>{}) : with_d(std::integral_constant<int, 128>{});
}

}  // namespace

cudaError_t configure_attn_dq() {
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < 8 && e == cudaSuccess; ++k)
        e = dispatch(k & 1 ? 64 : 128, k & 2 ? 1 : 2, (k & 4) != 0, [](auto d, auto t, auto causal) {
            constexpr int D = decltype(d)::value, kTiles = decltype(t)::value;
            constexpr bool kCausal = decltype(causal)::value;
            auto set = [](auto kernel) {
                return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, DqCfg<D, kTiles>::kSmemBytes);
            };
            cudaError_t r = set(attn_delta_kernel<D, kTiles, kCausal>);
            if constexpr (D == 128) {
                if (r == cudaSuccess) r = set(attn_dq_kernel<D, kTiles, kCausal, false>);
                if (r == cudaSuccess) r = set(attn_dq_kernel<D, kTiles, kCausal, true>);
            }
            return r;
        });
    return e;
}

cudaError_t launch_attn_dq(const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV,
                           const CUtensorMap& tmdO, const CUtensorMap& tmdQ, bool strided, uint32_t orders,
                           const float* LSE, const float* Delta, const AttnShape& s, int num_sms, int* dev_status,
                           cudaStream_t stream) {
    const Plan p = plan_of(s, num_sms);
    return dispatch(s.D, p.tiles, s.causal, [&](auto d, auto t, auto causal) {
        constexpr int D = decltype(d)::value, kTiles = decltype(t)::value;
        constexpr bool kCausal = decltype(causal)::value;
        if constexpr (D == 64) {
            return cudaErrorNotSupported;  // (attn_dq64.cu)
        } else {
            auto go = [&](auto kernel) {
                return launch_overlapped(kernel, p.grid, dim3(kThreads), DqCfg<D, kTiles>::kSmemBytes, stream, tmQ, tmK, tmV,
                                         tmdO, tmdQ, LSE, Delta, s.T, s.B * s.H, s.H, orders, p.n_blocks, p.chunk, s.scale,
                                         dev_status);
            };
            return strided ? go(attn_dq_kernel<D, kTiles, kCausal, true>) : go(attn_dq_kernel<D, kTiles, kCausal, false>);
        }
    });
}

cudaError_t launch_attn_delta(const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV,
                              const CUtensorMap& tmdO, const float* LSE, float* Delta, const AttnShape& s,
                              int num_sms, int* dev_status, cudaStream_t stream) {
    const Plan p = plan_of(s, num_sms);
    return dispatch(s.D, p.tiles, s.causal, [&](auto d, auto t, auto causal) {
        constexpr int D = decltype(d)::value, kTiles = decltype(t)::value;
        constexpr bool kCausal = decltype(causal)::value;
        return launch_overlapped(attn_delta_kernel<D, kTiles, kCausal>, p.grid, dim3(kThreads), DqCfg<D, kTiles>::kSmemBytes,
                                 stream, tmQ, tmK, tmV, tmdO, LSE, Delta, s.T, s.B * s.H, p.n_blocks, p.chunk, s.scale,
                                 dev_status);
    });
}

}  // namespace nova
