// Query-major passes of the backward at D = 64 (see attn_dq.cu for what they compute: dQ of the two-kernel backward, and the
// exact Delta), with the operands that an item keeps in tensor memory, as in attn_dkdv64.cu.
//
// A work item is one 128-row query tile of one head; its keys go by in steps of 64, which alternate between two compute
// groups:
//   S  = Q_i K_s^T,  dP = dO_i V_s^T          (Q_i and dO_i in tensor memory, K_s and V_s from smem)
//   P  = exp2(S*c - LSE*log2e),  dS = P * (dP - Delta)
//   dQ += dS K_s                              (dS as bf16 in tensor memory, K read MN-major), or Delta += P . dP
// What bounds it: 64 exponentials per thread and step, 1024 clocks of the exp2 unit per 128 x 128 block; the products take
// 768 with the A operands in tensor memory (1024 with all of them in shared memory, whose port a product of N = 64 then
// saturates).  S and dP run ahead of the compute groups: the columns of a step are handed back as soon as they have been
// read.  A step takes some 670 clocks, the end of an item 1300, a launch 10000 besides.  Under ncu (us), the pairs of tiles of
// attn_dq.cu and so: dQ at H=12, B=8, T=1024: 38, 33; B=4, T=1500: 37, 33; B=32, T=1024: 117, 103; B=1, T=8192: 189, 155; exact
// Delta: 32, 30; 32, 30; 98, 94; 163, 143.  Items are handed out dynamically (WorkRing), heaviest first.  512 threads:
//   warp 0      TMA producer: Q_i and dO_i double-buffered, K_s and V_s through a ring of 64-key stages
//   warps 1-3   UMMA issuers of S, dP and dQ (why three: see attn_dkdv64.cu)
//   warps 4-7   compute group 0, warps 8-11 group 1: a thread has one query row and the 64 keys of its step
//   warps 12-15 Q_i and dO_i from shared into tensor memory, the row terms, and dQ (or Delta) of a finished item out
// TMEM columns: dQ [0,64)  Q [64,96)  dO [96,128), then per group S 64, dP 64, two buffers of dS, 32 each.
#include "kernels.h"
#include "ptx.cuh"

namespace nova {
namespace {

constexpr int D = 64;
constexpr int kThreads = 512;
constexpr int kTmemCols = 512;
constexpr int kStep = kKeyStep;              // keys per step
constexpr int kStepBytes = kStep * 128;      // one [64 rows x 64 bf16] box
constexpr int kTileBytes = kHalfTileBytes;   // one [128 rows x 64 bf16] box
constexpr int kStages = 8;

constexpr int kOffQ = 0;                                 // [2]
constexpr int kOffdO = 2 * kTileBytes;                   // [2]
constexpr int kOffOut = 4 * kTileBytes;                  // dQ on its way out
constexpr int kOffK = 5 * kTileBytes;                    // [kStages]
constexpr int kOffV = kOffK + kStages * kStepBytes;      // [kStages]
constexpr int kOffRow = kOffV + kStages * kStepBytes;    // [2 items][128] of (-LSE*log2e, -Delta)
constexpr int kOffSum = kOffRow + 2 * kBlockQ * 8;       // [2 items][2 groups][128]: partial sums of Delta
constexpr int kOffBar = kOffSum + 4 * kBlockQ * 4;
constexpr int kSmemBytes = kOffBar + 512 + 1024;
static_assert(kSmemBytes <= 232448, "exceeds the shared memory of one CTA");
constexpr int kColdQ = 0, kColQ = 64, kColdO = 96;
constexpr int kColS = 128, kColdP = 192, kColdS = 256, kGroupCols = 192;  // + kGroupCols * group

struct Dq64Bars {
    uint64_t q_full[2], q_empty[2];
    uint64_t kv_full[kStages], kv_empty[kStages];
    uint64_t sp_full[2], s_free[2], dp_free[2];  // per group
    // by step & 3, i.e. two per group: a group may finish a step before the one before has been seen, and a single barrier
    // two phases on looks as if it had not moved
    uint64_t ready[4], ds_done[4];
    uint64_t op_full[2], op_free[2];             // Q, dO of an item in tensor memory; no longer read there
    // by item & 1: the compute groups may be in different items, and edge warps an item ahead
    uint64_t rows_full[2];                       // the row terms of an item are there
    uint64_t out_full[2], out_free;              // dQ (or the partial sums) of an item complete; read
    uint64_t staged, stage_free;                 // the edge warps among themselves
    uint64_t drain[3];
    WorkRing ring;
    uint32_t tmem_base;
    int abort_flag;
};
static_assert(sizeof(Dq64Bars) <= 512, "barrier block");

// Work items: 128-row query tiles, heaviest first (the last tile of a causal problem sees every key).
struct Dq64Work {
    int BH, n_tiles, T, H;
    uint32_t orders;  // coordinate orders of the Q, K, V, dO, dQ tensor maps, four bits each
    bool causal;
    // Query tile, head and number of key steps of item `idx`.
    __device__ __forceinline__ void get(int idx, int* qt, int* bh, int* n) const {
        const int order = idx / BH;
        *qt = n_tiles - 1 - order;
        *bh = idx - order * BH;
        const int n_all = (T + kStep - 1) / kStep;
        *n = causal ? min((*qt + 1) * (kBlockQ / kStep), n_all) : n_all;
    }
};

template <bool kStrided>
__device__ __forceinline__ void dq64_producer(const CUtensorMap* tmQ, const CUtensorMap* tmK, const CUtensorMap* tmV,
                                              const CUtensorMap* tmdO, uint8_t* smem, Dq64Bars* bars, const Dq64Work& wk) {
    volatile int* abort_flag = &bars->abort_flag;
    bool ok = true, clc_pending = false;
    int w = 0, n_q = 0, g = 0, st = 0;  // items, Q and dO requested; steps requested
    uint32_t ph = 0;
    int item = blockIdx.x;
    for (;;) {
        if (w > 0) ok = bars->ring.publish(w, item, abort_flag, kWaitLimitCycles);
        if (!ok || item < 0) break;
        int qt, bh, n;
        wk.get(item, &qt, &bh, &n);
        if (w == 0) griddep_wait();
        const int head = kStrided ? bh % wk.H : 0, batch = kStrided ? bh / wk.H : 0;
        const int qs = w & 1;
        ok = mbar_wait(&bars->q_empty[qs], ((w >> 1) & 1) ^ 1, abort_flag);
        if (!ok) break;
        mbar_expect_tx(&bars->q_full[qs], 2 * kTileBytes);  // rows past T arrive as zeros
        ++n_q;
        tma_load_tile<kStrided>(smem + kOffQ + qs * kTileBytes, tmQ, &bars->q_full[qs], wk.orders & 15, 0, qt * kBlockQ, head,
                                batch, bh);
        tma_load_tile<kStrided>(smem + kOffdO + qs * kTileBytes, tmdO, &bars->q_full[qs], (wk.orders >> 12) & 15, 0,
                                qt * kBlockQ, head, batch, bh);
        for (int s = 0; s < n; ++s) {
            ok = mbar_wait(&bars->kv_empty[st], ph ^ 1, abort_flag);
            if (!ok) break;
            mbar_expect_tx(&bars->kv_full[st], 2 * kStepBytes);
            ++g;
            tma_load_tile<kStrided>(smem + kOffK + st * kStepBytes, tmK, &bars->kv_full[st], (wk.orders >> 4) & 15, 0, s * kStep,
                                    head, batch, bh);
            tma_load_tile<kStrided>(smem + kOffV + st * kStepBytes, tmV, &bars->kv_full[st], (wk.orders >> 8) & 15, 0, s * kStep,
                                    head, batch, bh);
            if (++st == kStages) {
                st = 0;
                ph ^= 1;
            }
        }
        if (!ok) break;
        // all loads of this item are on their way: claim the next one now, and no earlier
        bars->ring.request();
        clc_pending = true;
        ok = bars->ring.answer(w, &item, abort_flag, kWaitLimitCycles);
        if (!ok) break;
        clc_pending = false;
        ++w;
    }
    if (!ok) {  // giving up: let what is in flight land before the CTA's shared memory goes away
        int none = 0;
        if (clc_pending) (void)mbar_wait(&bars->ring.answer_bar, w & 1, &none);
        for (int x = n_q > 2 ? n_q - 2 : 0; x < n_q; ++x) (void)mbar_wait(&bars->q_full[x & 1], (x >> 1) & 1, &none);
        for (int x = g > kStages ? g - kStages : 0; x < g; ++x)
            (void)mbar_wait(&bars->kv_full[x % kStages], (x / kStages) & 1, &none);
    }
}

// S (kdP false) and dP (kdP true) of each step, as soon as the compute group has read those of its last step.  dP waits for
// dQ of the group's last but one step besides, so that a group that sees both finds its buffer of dS free.
template <bool kdP, bool kDelta>
__device__ __forceinline__ void dq64_mma_sp(uint8_t* smem, Dq64Bars* bars, uint32_t tmem_base, const Dq64Work& wk) {
    volatile int* abort_flag = &bars->abort_flag;
    constexpr uint32_t kIdescT = umma_idesc_bf16(128, kStep, 0, 0);
    const uint32_t hi = umma_desc_hi_sw128(1024);
    const uint32_t b0 = umma_desc_lo(smem_u32(smem + (kdP ? kOffV : kOffK)), 16);
    const bool el = elect_one();
    const int lane = threadIdx.x & 31;
    bool ok = true;
    int g = 0, st = 0;
    uint32_t ph = 0;
    for (int w = 0;; ++w) {
        const int item = bars->ring.take(w, lane, abort_flag, kWaitLimitCycles);
        if (item < 0) {
            ok = (item == -1);
            break;
        }
        int qt, bh, n;
        wk.get(item, &qt, &bh, &n);
        if (w == 0) griddep_wait();
        ok = mbar_wait(&bars->op_full[kdP], w & 1, abort_flag);
        if (!ok) break;
        for (int s = 0; s < n; ++s, ++g) {
            ok = mbar_wait(&bars->kv_full[st], ph, abort_flag);
            if (ok) ok = mbar_wait(kdP ? &bars->dp_free[g & 1] : &bars->s_free[g & 1], ((g >> 1) & 1) ^ 1, abort_flag);
            if (ok && kdP && !kDelta) ok = mbar_wait(&bars->ds_done[g & 3], ((g >> 2) & 1) ^ 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            if (el) {
                const uint32_t t_acc = tmem_base + (kdP ? kColdP : kColS) + kGroupCols * (g & 1);
                const uint32_t b = b0 + st * (kStepBytes >> 4);
#pragma unroll
                for (int k = 0; k < D / 16; ++k)
                    umma_ts(t_acc, tmem_base + (kdP ? kColdO : kColQ) + 8 * k, umma_desc_join(b + 2 * k, hi), kIdescT,
                            k > 0 ? 1u : 0u);
                tc_commit(&bars->sp_full[g & 1]);
                if (kDelta) tc_commit(&bars->kv_empty[st]);
                if (s + 1 == n) tc_commit(&bars->op_free[kdP]);
            }
            __syncwarp();
            if (++st == kStages) {
                st = 0;
                ph ^= 1;
            }
        }
        if (!ok) break;
    }
    if (!ok) {
        int none = 0;
        if (el) tc_commit(&bars->drain[kdP]);
        __syncwarp();
        (void)mbar_wait(&bars->drain[kdP], 0, &none);
    }
}

// dQ of each step, in key order.
__device__ __forceinline__ void dq64_mma_dq(uint8_t* smem, Dq64Bars* bars, uint32_t tmem_base, const Dq64Work& wk) {
    volatile int* abort_flag = &bars->abort_flag;
    constexpr uint32_t kIdescdQ = umma_idesc_bf16(128, D, 0, 1);  // A from TMEM, B (K) MN-major
    const uint32_t hi = umma_desc_hi_sw128(1024);
    const uint32_t k_m0 = umma_desc_lo(smem_u32(smem + kOffK), kStepBytes);
    const bool el = elect_one();
    const int lane = threadIdx.x & 31;
    bool ok = true;
    int g = 0, st = 0;
    for (int w = 0;; ++w) {
        const int item = bars->ring.take(w, lane, abort_flag, kWaitLimitCycles);
        if (item < 0) {
            ok = (item == -1);
            break;
        }
        int qt, bh, n;
        wk.get(item, &qt, &bh, &n);
        if (w == 0) {
            griddep_wait();
            if (el) griddep_launch_dependents();  // the dK/dV kernel, which needs nothing of dQ, but what was there before (ptx.cuh)
            __syncwarp();
        }
        // the previous item's dQ must have been read out of TMEM before it is overwritten
        if (w > 0) ok = mbar_wait(&bars->out_free, (w - 1) & 1, abort_flag);
        if (!ok) break;
        for (int s = 0; s < n; ++s, ++g) {
            ok = mbar_wait(&bars->ready[g & 3], (g >> 2) & 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            if (el) {
                const uint32_t t_ds = tmem_base + kColdS + kGroupCols * (g & 1) + 32 * ((g >> 1) & 1);
                const uint32_t b = k_m0 + st * (kStepBytes >> 4);
#pragma unroll
                for (int k = 0; k < kStep / 16; ++k)  // 16 keys: 8 packed columns, 16 smem rows = 2048 bytes
                    umma_ts(tmem_base + kColdQ, t_ds + k * 8, umma_desc_join(b + k * 128, hi), kIdescdQ,
                            (s > 0 || k > 0) ? 1u : 0u);
                tc_commit(&bars->ds_done[g & 3]);
                tc_commit(&bars->kv_empty[st]);
                if (s + 1 == n) tc_commit(&bars->out_full[w & 1]);
            }
            __syncwarp();
            if (++st == kStages) st = 0;
        }
        if (!ok) break;
    }
    if (!ok) {
        int none = 0;
        if (el) tc_commit(&bars->drain[2]);
        __syncwarp();
        (void)mbar_wait(&bars->drain[2], 0, &none);
    }
}

// Compute group `grp` (steps g with g % 2 == grp), warp `cwarp` of it.
template <bool kCausal, bool kDelta>
__device__ __forceinline__ void dq64_compute(uint8_t* smem, Dq64Bars* bars, uint32_t tmem_base, float scale, const Dq64Work& wk,
                                             int grp, int cwarp, int lane) {
    volatile int* abort_flag = &bars->abort_flag;
    const uint32_t lane_base = 32u * cwarp;
    const int r = lane_base + lane;  // local query row
    const float c = scale * kLog2e;
    const uint64_t c2 = f32x2_pack(c, c);
    const uint32_t t_s = tmem_addr(tmem_base, lane_base, kColS + kGroupCols * grp);
    const uint32_t t_dp = t_s + (kColdP - kColS), t_ds = t_s + (kColdS - kColS);
    bool ok = true;
    int g = 0;         // steps of all items so far
    uint32_t k = 0;    // steps of this group

    for (int w = 0;; ++w) {
        const int item = bars->ring.take(w, lane, abort_flag, kWaitLimitCycles);
        if (item < 0) {
            ok = (item == -1);
            break;
        }
        int qt, bh, n;
        wk.get(item, &qt, &bh, &n);
        if (w == 0) griddep_wait();
        ok = mbar_wait(&bars->rows_full[w & 1], (w >> 1) & 1, abort_flag);
        if (!ok) break;
        const float2 row_terms = reinterpret_cast<const float2*>(smem + kOffRow)[(w & 1) * kBlockQ + r];
        const uint64_t nlse = f32x2_pack(row_terms.x, row_terms.x), nd = f32x2_pack(row_terms.y, row_terms.y);
        const int row = qt * kBlockQ + r;
        uint64_t acc0 = 0, acc1 = 0;
        for (int s = (g ^ grp) & 1; s < n; s += 2, ++k) {
            ok = mbar_wait(&bars->sp_full[grp], k & 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            uint32_t pf[kStep];
            tmem_ld_x32(t_s, pf);
            tmem_ld_x32(t_s + 32, pf + 32);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->s_free[grp]);
            // Mask from indices only: causal keeps key <= query, the end of the sequence key < T.
            const int lim = (kCausal ? min(row, wk.T - 1) : wk.T - 1) - s * kStep;  // last kept key of the step
            if ((kCausal && (s + 1) * kStep > qt * kBlockQ) || (s + 1) * kStep > wk.T) {
#pragma unroll
                for (int i = 0; i < kStep; ++i)
                    if (i > lim) pf[i] = 0xff800000u;  // -inf: P = 0
            }
#pragma unroll
            for (int i = 0; i < kStep; i += 2) {
                float x0, x1;
                f32x2_unpack(f32x2_fma(f32x2_pack(__uint_as_float(pf[i]), __uint_as_float(pf[i + 1])), c2, nlse), x0, x1);
                pf[i] = __float_as_uint(ex2_approx(x0));
                pf[i + 1] = __float_as_uint(ex2_approx(x1));
            }
            // dP 16 keys at a time
            uint32_t dv[16];
            tmem_ld_x16(t_dp, dv);
#pragma unroll
            for (int x = 0; x < kStep; x += 16) {
                tmem_wait_ld();
                uint32_t dd[8];
#pragma unroll
                for (int y = 0; y < 8; ++y) {
                    const uint64_t p = f32x2_pack(__uint_as_float(pf[x + 2 * y]), __uint_as_float(pf[x + 2 * y + 1]));
                    const uint64_t e = f32x2_pack(__uint_as_float(dv[2 * y]), __uint_as_float(dv[2 * y + 1]));
                    if constexpr (kDelta) {
                        uint64_t& acc = (y & 1) ? acc1 : acc0;
                        acc = f32x2_fma(p, e, acc);
                    } else {
                        float d0, d1;
                        f32x2_unpack(f32x2_mul(p, f32x2_add(e, nd)), d0, d1);
                        dd[y] = pack_bf16x2(d0, d1);
                    }
                }
                if (x + 16 < kStep) {
                    tmem_ld_x16(t_dp + x + 16, dv);
                } else {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bars->dp_free[grp]);
                }
                if constexpr (!kDelta) tmem_st_x8(t_ds + 32 * (k & 1) + x / 2, dd);
            }
            if constexpr (!kDelta) {
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars->ready[grp + 2 * (k & 1)]);
            }
        }
        if (!ok) break;
        if constexpr (kDelta) {
            float a0, a1, a2, a3;
            f32x2_unpack(acc0, a0, a1);
            f32x2_unpack(acc1, a2, a3);
            reinterpret_cast<float*>(smem + kOffSum)[((w & 1) * 2 + grp) * kBlockQ + r] = (a0 + a1) + (a2 + a3);
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->out_full[w & 1]);
        }
        g += n;
    }
}

// Edge warps (warp `ow` of four, thread = query row): Q and dO of an item from shared into tensor memory, each as soon as the
// last product that reads these columns is done, and the row terms; then dQ * scale of the item before as bf16 into
// shared memory and out with a TMA store, or its Delta.
template <bool kStrided, bool kDelta>
__device__ __forceinline__ void dq64_edges(uint8_t* smem, Dq64Bars* bars, uint32_t tmem_base, const CUtensorMap* tmdQ,
                                           const float* __restrict__ LSE, const float* __restrict__ Delta,
                                           float* __restrict__ Delta_out, float scale, const Dq64Work& wk, int ow, int lane) {
    volatile int* abort_flag = &bars->abort_flag;
    const uint32_t lane_base = 32u * ow;
    const int r = lane_base + lane;
    const bool leader = (ow == 0 && lane == 0);
    bool ok = true;

    // Q (v = 0) or dO (v = 1) of the w-th item: a row of 64 bf16 numbers is 32 columns
    auto operand = [&](int w, int v) -> bool {
        const int qs = w & 1;
        if (v == 0 && !mbar_wait(&bars->q_full[qs], (w >> 1) & 1, abort_flag)) return false;
        uint32_t a[32];
#pragma unroll
        for (int ch = 0; ch < 8; ++ch) {
            const uint4 x = *reinterpret_cast<const uint4*>(smem + (v ? kOffdO : kOffQ) + qs * kTileBytes + r * 128 +
                                                            ((ch ^ (r & 7)) << 4));
            a[4 * ch] = x.x, a[4 * ch + 1] = x.y, a[4 * ch + 2] = x.z, a[4 * ch + 3] = x.w;
        }
        if (w > 0 && !mbar_wait(&bars->op_free[v], (w - 1) & 1, abort_flag)) return false;
        tc_fence_after();
        __syncwarp();
        tmem_st_x32(tmem_addr(tmem_base, lane_base, v ? kColdO : kColQ), a);
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
            if (v == 1) mbar_arrive(&bars->q_empty[qs]);
            mbar_arrive(&bars->op_full[v]);
        }
        return true;
    };
    auto write_out = [&](int w, int qt, int bh) -> bool {
        if (!mbar_wait(&bars->out_full[w & 1], (w >> 1) & 1, abort_flag)) return false;
        if constexpr (kDelta) {
            // even steps, odd steps: the order in which attn_dq.cu sums them at D=64, too
            const float* sum = reinterpret_cast<const float*>(smem + kOffSum) + (w & 1) * 2 * kBlockQ;
            const int row = qt * kBlockQ + r;
            if (row < wk.T) Delta_out[static_cast<size_t>(bh) * wk.T + row] = sum[r] + sum[kBlockQ + r];
            return true;
        }
        tc_fence_after();
        __syncwarp();
        uint32_t pk[32];
#pragma unroll
        for (int cb = 0; cb < D; cb += 32) {
            uint32_t a[32];
            tmem_ld_x32(tmem_addr(tmem_base, lane_base, kColdQ + cb), a);
            tmem_wait_ld();
#pragma unroll
            for (int x = 0; x < 16; ++x)
                pk[cb / 2 + x] = pack_bf16x2(__uint_as_float(a[2 * x]) * scale, __uint_as_float(a[2 * x + 1]) * scale);
        }
        tc_fence_before();
        if (leader) {  // the buffer is free once what was sent from it last has been read
            bulk_wait_group_read<0>();
            mbar_arrive(&bars->stage_free);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->out_free);
        if (!mbar_wait(&bars->stage_free, w & 1, abort_flag)) return false;
#pragma unroll
        for (int x = 0; x < 8; ++x)
            *reinterpret_cast<uint4*>(smem + kOffOut + r * 128 + ((x ^ (r & 7)) << 4)) =
                make_uint4(pk[4 * x], pk[4 * x + 1], pk[4 * x + 2], pk[4 * x + 3]);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->staged);
        bool leader_ok = true;
        if (leader) {
            leader_ok = mbar_wait(&bars->staged, w & 1, abort_flag);
            if (leader_ok) {
                tma_store_tile<kStrided>(tmdQ, smem + kOffOut, (wk.orders >> 16) & 15, 0, qt * kBlockQ,
                                         kStrided ? bh % wk.H : 0, kStrided ? bh / wk.H : 0, bh);
                bulk_commit_group();
            }
        }
        return __all_sync(0xffffffffu, leader_ok);
    };

    int qt_out = 0, bh_out = 0;
    for (int w = 0; ok; ++w) {
        const int item = bars->ring.take(w, lane, abort_flag, kWaitLimitCycles);
        if (item < 0) {
            if (item == -1 && w > 0) (void)write_out(w - 1, qt_out, bh_out);
            break;
        }
        int qt, bh, n;
        wk.get(item, &qt, &bh, &n);
        if (w == 0) griddep_wait();
        // Rows past the end of the sequence: LSE = +inf gives P = 0 everywhere.
        const int row = qt * kBlockQ + r;
        const size_t idx = static_cast<size_t>(bh) * wk.T + row;
        float2 terms = make_float2(row < wk.T ? -LSE[idx] * kLog2e : -INFINITY, 0.f);
        if (!kDelta && row < wk.T) terms.y = -Delta[idx];
        ok = operand(w, 0);
        if (ok) ok = operand(w, 1);
        if (!ok) break;
        // (the compute groups have been through the item before the last: its dQ or its sums were complete)
        reinterpret_cast<float2*>(smem + kOffRow)[(w & 1) * kBlockQ + r] = terms;
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->rows_full[w & 1]);
        if (w > 0) ok = write_out(w - 1, qt_out, bh_out);
        qt_out = qt;
        bh_out = bh;
    }
    if (!kDelta && leader) bulk_wait_group<0>();  // dQ must be complete before the kernel ends
}

template <bool kCausal, bool kStrided, bool kDelta>
__device__ __forceinline__ void dq64_body(const CUtensorMap* tmQ, const CUtensorMap* tmK, const CUtensorMap* tmV,
                                          const CUtensorMap* tmdO, const CUtensorMap* tmdQ, const float* __restrict__ LSE,
                                          const float* __restrict__ Delta, float* __restrict__ Delta_out, const Dq64Work& wk,
                                          float scale, int* __restrict__ dev_status) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    Dq64Bars* bars = reinterpret_cast<Dq64Bars*>(smem + kOffBar);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(&bars->q_full[s], 1);
            mbar_init(&bars->q_empty[s], 4);
            mbar_init(&bars->sp_full[s], 2);  // S and dP
            mbar_init(&bars->s_free[s], 4);
            mbar_init(&bars->dp_free[s], 4);
            mbar_init(&bars->op_full[s], 4);
            mbar_init(&bars->op_free[s], 1);
            mbar_init(&bars->rows_full[s], 4);
            mbar_init(&bars->out_full[s], kDelta ? 8 : 1);
        }
        for (int s = 0; s < 4; ++s) {
            mbar_init(&bars->ready[s], 4);
            mbar_init(&bars->ds_done[s], 1);
        }
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&bars->kv_full[s], 1);
            mbar_init(&bars->kv_empty[s], kDelta ? 2 : 1);  // S and dP, or dQ, which comes after both
        }
        mbar_init(&bars->out_free, 4);
        mbar_init(&bars->staged, 4);
        mbar_init(&bars->stage_free, 1);
        for (int s = 0; s < 3; ++s) mbar_init(&bars->drain[s], 1);
        bars->ring.init((kDelta ? 2 : 3) + 8 + 4);  // issuers, compute warps, edge warps
        bars->ring.publish_first(blockIdx.x);
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
    if (kDelta) griddep_launch_dependents();
    // Everything above overlaps the previous kernel of the stream, and so does finding out what the first item is: with the wait
    // here instead, forward, exact Delta and backward of H=148, T=192 took 27.0 us, not 26.2.  Every role waits then, those
    // that touch no global memory too: they would wait for the others on barriers, whose waits are bounded, while the previous
    // kernel may take as long as it likes.

    if (warp == 0) {
        if (lane == 0) dq64_producer<kStrided>(tmQ, tmK, tmV, tmdO, smem, bars, wk);
    } else if (warp == 1) {
        dq64_mma_sp<false, kDelta>(smem, bars, tmem_base, wk);
    } else if (warp == 2) {
        dq64_mma_sp<true, kDelta>(smem, bars, tmem_base, wk);
    } else if (warp == 3) {
        if constexpr (!kDelta) dq64_mma_dq(smem, bars, tmem_base, wk);
    } else if (warp >= 12) {
        dq64_edges<kStrided, kDelta>(smem, bars, tmem_base, tmdQ, LSE, Delta, Delta_out, scale, wk, warp & 3, lane);
    } else {
        dq64_compute<kCausal, kDelta>(smem, bars, tmem_base, scale, wk, (warp - 4) >> 2, warp & 3, lane);
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, kTmemCols);
    if (threadIdx.x == 0 && bars->abort_flag != 0) atomicExch(dev_status, kDevTimeout);
}

template <bool kCausal, bool kStrided>
__global__ void __launch_bounds__(kThreads, 1)
attn_dq64_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                 const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmdO,
                 const __grid_constant__ CUtensorMap tmdQ, const float* __restrict__ LSE, const float* __restrict__ Delta, int T,
                 int BH, int H, uint32_t orders, int n_tiles, float scale, int* __restrict__ dev_status) {
    dq64_body<kCausal, kStrided, false>(&tmQ, &tmK, &tmV, &tmdO, &tmdQ, LSE, Delta, nullptr,
                                        Dq64Work{BH, n_tiles, T, H, orders, kCausal}, scale, dev_status);
}

template <bool kCausal>
__global__ void __launch_bounds__(kThreads, 1)
attn_delta64_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                    const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmdO,
                    const float* __restrict__ LSE, float* __restrict__ Delta, int T, int BH, int n_tiles, float scale,
                    int* __restrict__ dev_status) {
    dq64_body<kCausal, false, true>(&tmQ, &tmK, &tmV, &tmdO, nullptr, LSE, nullptr, Delta,
                                    Dq64Work{BH, n_tiles, T, 1, 0u, kCausal}, scale, dev_status);
}

}  // namespace

cudaError_t configure_attn_dq64() {
    auto set = [](auto kernel) {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    };
    cudaError_t e = set(attn_dq64_kernel<true, false>);
    if (e == cudaSuccess) e = set(attn_dq64_kernel<true, true>);
    if (e == cudaSuccess) e = set(attn_dq64_kernel<false, false>);
    if (e == cudaSuccess) e = set(attn_dq64_kernel<false, true>);
    if (e == cudaSuccess) e = set(attn_delta64_kernel<true>);
    if (e == cudaSuccess) e = set(attn_delta64_kernel<false>);
    return e;
}

cudaError_t launch_attn_dq64(const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV,
                             const CUtensorMap& tmdO, const CUtensorMap& tmdQ, bool strided, uint32_t orders,
                             const float* LSE, const float* Delta, const AttnShape& s, int* dev_status, cudaStream_t stream) {
    const int n_tiles = (s.T + kBlockQ - 1) / kBlockQ, BH = s.B * s.H;
    const dim3 grid(static_cast<unsigned>(n_tiles) * BH);  // one CTA per item; those that do not start are taken over
    auto go = [&](auto kernel) {
        return launch_overlapped(kernel, grid, dim3(kThreads), kSmemBytes, stream, tmQ, tmK, tmV, tmdO, tmdQ, LSE, Delta, s.T, BH,
                                 s.H, orders, n_tiles, s.scale, dev_status);
    };
    if (s.causal) return strided ? go(attn_dq64_kernel<true, true>) : go(attn_dq64_kernel<true, false>);
    return strided ? go(attn_dq64_kernel<false, true>) : go(attn_dq64_kernel<false, false>);
}

cudaError_t launch_attn_delta64(const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV,
                                const CUtensorMap& tmdO, const float* LSE, float* Delta, const AttnShape& s, int* dev_status,
                                cudaStream_t stream) {
    const int n_tiles = (s.T + kBlockQ - 1) / kBlockQ, BH = s.B * s.H;
    const dim3 grid(static_cast<unsigned>(n_tiles) * BH);
    auto go = [&](auto kernel) {
        return launch_overlapped(kernel, grid, dim3(kThreads), kSmemBytes, stream, tmQ, tmK, tmV, tmdO, LSE, Delta, s.T, BH,
                                 n_tiles, s.scale, dev_status);
    };
    return s.causal ? go(attn_delta64_kernel<true>) : go(attn_delta64_kernel<false>);
}

}  // namespace nova
