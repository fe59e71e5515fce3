// dK and dV of the two-kernel backward at D = 64 (paper Section 4.2, "The Backward Pass": one kernel reduces dQ over
// keys, the other reduces dK and dV over queries; the probability matrix is rebuilt from the saved log-sum-exp, never
// stored; the causal loop bound is raised so that queries above the diagonal are never visited).
//
// A work item is one 128-key tile of one head; its queries go by in steps of 64, which alternate between two compute
// groups.  Everything is transposed, keys on the lanes of tensor memory:
//   S^T  = K_j Q_s^T - LSE_s/scale,  dP^T = V_j dO_s^T - Delta_s   (K_j and V_j in tensor memory, the rest from smem)
//   P^T  = exp2(S^T*c),  dS^T = P^T * dP^T                         (bf16, back into tensor memory)
//   dV  += P^T dO_s,  dK += dS^T Q_s                               (tensor memory x smem, dO and Q read MN-major)
// K_j and V_j are A operands in tensor memory, put there once per item: a product of M=128, N=64 with both operands in
// shared memory takes 48 clocks per 16 k elements, 6 KB through the one 128-byte port; with A in tensor memory it takes
// the 32 clocks of the arithmetic, and leaves three quarters of the port to the other users.
// What bounds it: a step takes 608 clocks of the tensor pipe (of which the row terms 96), 512 of the exp2 unit and some 780 in
// all, the rest being the chain dS^T -> dK -> dP^T of a group; the end of an item costs 2000 clocks, a launch 10000 besides
// (fitted to three of the shapes below), so that at T=1024, with nine steps an item, a step comes to 1200 of its SM's clocks.
// dK and dV under ncu (us), with the fused kernel without its dQ product and so: H=12, B=8, T=1024: 52, 38; B=4, T=1500:
// 53, 38; B=32, T=1024: 183, 125; B=1, T=8192: 286, 182; B=8, T=512: 22, 18.
// All 128 registers that 512 threads may have are in use, and 64 bytes of stack besides (56 where the kernel makes the row
// terms itself; 76 and 68 bytes of spill stores, 156 and 108 of loads in the code).
// Items are handed out dynamically (WorkRing), heaviest first.  512 threads:
//   warp 0      TMA producer: K_j and V_j double-buffered, Q_s and dO_s through a ring of 64-query stages
//   warps 1-3   UMMA issuers of S^T, of dP^T, and of dV and dK
//   warps 4-7   compute group 0, warps 8-11 group 1; a thread has one key row and the 64 queries of its step
//   warps 12-15 K_j and V_j from shared into tensor memory; -LSE/scale and -Delta of each step as operands of the products;
//               dV and dK of a finished item out with TMA stores, while the compute warps are in the next item
// TMEM columns: dV [0,64)  dK [64,128)  K [128,160)  V [160,192), then per group S^T 64, dP^T / dS^T 64, P^T 32.
#include "kernels.h"
#include "ptx.cuh"

namespace nova {
namespace {

constexpr int D = 64;
constexpr int kThreads = 512;
constexpr int kTmemCols = 512;
constexpr int kStep = kKeyStep;              // queries per step
constexpr int kStepBytes = kStep * 128;      // one [64 rows x 64 bf16] box
constexpr int kTileBytes = kHalfTileBytes;   // one [128 rows x 64 bf16] box
constexpr int kQStages = 6;
constexpr int kWorkConsumers = 3 + 8 + 4;  // issuers, compute warps, write-out warps

constexpr int kOffK = 0;                                 // [2]
constexpr int kOffV = 2 * kTileBytes;                    // [2]
constexpr int kOffOut = 4 * kTileBytes;                  // dV, dK on their way out
constexpr int kOffQ = 6 * kTileBytes;                    // [kQStages]
constexpr int kOffdO = kOffQ + kQStages * kStepBytes;    // [kQStages]
// Row terms: operands of 16 columns, unswizzled: core matrices of 8 rows x 8 columns (128 bytes), the two of 8 rows
// adjacent.  Queries: -LSE/scale in columns 0, 2, 4, -Delta in 1, 3, 5, each as three bf16 numbers that add up to it to 24
// bits; the sign of a Delta that is not finite in 8.  The constants (128 rows) pick the one or the other.
constexpr int kExtCore = 128;
constexpr int kExtStep = kStep / 8 * 2 * kExtCore;
constexpr int kExtConst = 128 / 8 * 2 * kExtCore;
constexpr int kOffExt = kOffdO + kQStages * kStepBytes;  // [kQStages], then the constants for S^T and dP^T
constexpr int kExtBytes = kQStages * kExtStep + 2 * kExtConst;
constexpr int kOffBar = kOffExt + kExtBytes;
constexpr int kSmemBytes = kOffBar + 512 + 1024;
static_assert(kSmemBytes <= 232448, "exceeds the shared memory of one CTA");
constexpr int kColdV = 0, kColdK = 64, kColK = 128, kColV = 160;
constexpr int kColS = 192, kColdP = 256, kColP = 320, kGroupCols = 160;  // + kGroupCols * group

struct Kv64Bars {
    uint64_t kv_full[2], kv_empty[2];
    uint64_t q_full[kQStages], q_empty[kQStages];  // Q, dO and row terms of a step
    uint64_t s_full[2], s_free[2], dp_full[2], ready[2], ds_done[2];  // per group
    uint64_t op_full[2], op_free[2];      // K, V of an item in tensor memory; no longer read there
    uint64_t dkv_full, dkv_free;          // dV and dK of an item complete; read out of TMEM
    uint64_t staged, stage_free;          // the write-out warps among themselves
    uint64_t drain[3];
    StepRing ring;
    int odd_rows[kQStages];  // the stage's row terms hold a Delta that is not finite
    int rows_of[kQStages];   // 1 + the step whose row terms the edge warps have put into the stage last
    int asked_items, asked_steps, asked_clc;  // what the producer has asked for: loads of items, of steps; answers of the ring
    uint32_t tmem_base;
    int abort_flag;
};
static_assert(sizeof(Kv64Bars) <= 512, "barrier block");

// Work items: 128-key tiles, heaviest (first) tiles first.
struct Kv64Work {
    int BH, T, H;
    uint32_t orders;  // coordinate orders of the Q, K, V, dO, dK, dV tensor maps, four bits each
    bool causal;
    // Key tile, head, first step and number of steps of item `idx`.
    __device__ __forceinline__ void get(int idx, int* kt, int* bh, int* s0, int* n) const {
        *kt = idx / BH;
        *bh = idx - *kt * BH;
        *s0 = causal ? *kt * (kBlockK / kStep) : 0;
        *n = (T + kStep - 1) / kStep - *s0;
    }
};

// The operand row of one query: 16 columns in two halves of 16 bytes.
// LSE/scale is held below kMostLse, which keeps what an infinite LSE means (P = 0 for +inf, P = inf for -inf) without an
// infinity that would meet another in the sum; queries past the end of the sequence count as +inf.  A NaN becomes P = inf where
// the query is kept.  A Delta that is not finite must not reach S^T (0 * inf is NaN): it enters as kMostLse in a column of its
// own, times kMostLse for dP^T (infinite, for a NaN as well) and times 0 for S^T.
struct RowTerms {
    uint4 first, second;
    bool odd;  // the second half is not zero
};
__device__ __forceinline__ RowTerms row_terms(float l, float d) {
    RowTerms t;
    float odd = 0.f;
    if (!(fabsf(l) <= kMostLse)) l = l < 0.f ? -kMostLse : kMostLse;
    t.odd = !(fabsf(d) <= kMostLse);
    if (t.odd) {
        odd = copysignf(kMostLse, d);
        d = 0.f;
    }
    t.first = split_bf16x3(l, d);
    t.second = make_uint4(__bfloat16_as_ushort(__float2bfloat16_rn(odd)), 0u, 0u, 0u);
    return t;
}

// The row terms of every step of every head, laid out as the kernel's stages hold them: once per row instead of once per row
// and key tile, for callers that have room for them.
__global__ void __launch_bounds__(256) row_terms64_kernel(const float* __restrict__ LSE, const float* __restrict__ Delta,
                                                          uint8_t* __restrict__ terms, int T, int n_steps, long long rows,
                                                          float inv_scale) {
    griddep_launch_dependents();
    griddep_wait();
    const long long idx = static_cast<long long>(blockIdx.x) * 256 + threadIdx.x;
    if (idx >= rows) return;
    const uint32_t tile = static_cast<uint32_t>(idx / kStep), r = static_cast<uint32_t>(idx % kStep);
    const uint32_t bh = tile / n_steps, q = (tile - bh * n_steps) * kStep + r;
    const bool in = q < static_cast<uint32_t>(T);
    const size_t at = static_cast<size_t>(bh) * T + q;
    const RowTerms t = row_terms(in ? -LSE[at] * inv_scale : -kMostLse, in ? -Delta[at] : 0.f);
    uint8_t* const row = terms + static_cast<size_t>(tile) * kExtStep + (r >> 3) * 2 * kExtCore + (r & 7) * 16;
    *reinterpret_cast<uint4*>(row) = t.first;
    *reinterpret_cast<uint4*>(row + kExtCore) = t.second;
}

template <bool kStrided, bool kTerms>
__device__ __forceinline__ void kv64_producer(const CUtensorMap* tmQ, const CUtensorMap* tmK, const CUtensorMap* tmV,
                                              const CUtensorMap* tmdO, const uint8_t* __restrict__ terms, uint8_t* smem,
                                              Kv64Bars* bars, const Kv64Work& wk) {
    volatile int* abort_flag = &bars->abort_flag;
    bool ok = true;
    int w = 0, n_kv = 0, n_clc = 0, g = 0, st = 0;  // items; K and V, answers, steps requested
    uint32_t ph = 0;
    int item = blockIdx.x;
    for (;;) {
        int kt = 0, bh = 0, s0 = 0, n = -1;
        if (item >= 0) wk.get(item, &kt, &bh, &s0, &n);
        ok = bars->ring.publish_steps(w, item, n, abort_flag);
        if (!ok || item < 0) break;
        const int head = kStrided ? bh % wk.H : 0, batch = kStrided ? bh / wk.H : 0;
        const int ks = w & 1;
        ok = mbar_wait(&bars->kv_empty[ks], ((w >> 1) & 1) ^ 1, abort_flag);
        if (!ok) break;
        mbar_expect_tx(&bars->kv_full[ks], 2 * kTileBytes);  // rows past T arrive as zeros
        ++n_kv;
        tma_load_tile<kStrided>(smem + kOffK + ks * kTileBytes, tmK, &bars->kv_full[ks], (wk.orders >> 4) & 15, 0,
                                kt * kBlockK, head, batch, bh);
        tma_load_tile<kStrided>(smem + kOffV + ks * kTileBytes, tmV, &bars->kv_full[ks], (wk.orders >> 8) & 15, 0,
                                kt * kBlockK, head, batch, bh);
        for (int s = 0; s < n; ++s) {
            ok = mbar_wait(&bars->q_empty[st], ph ^ 1, abort_flag);
            if (!ok) break;
            mbar_expect_tx(&bars->q_full[st], 2 * kStepBytes + (kTerms ? kExtStep : 0));
            ++g;
            if (kTerms)
                bulk_load(smem + kOffExt + st * kExtStep,
                          terms + (static_cast<size_t>(bh) * ((wk.T + kStep - 1) / kStep) + s0 + s) * kExtStep, kExtStep,
                          &bars->q_full[st]);
            tma_load_tile<kStrided>(smem + kOffQ + st * kStepBytes, tmQ, &bars->q_full[st], wk.orders & 15, 0,
                                    (s0 + s) * kStep, head, batch, bh);
            tma_load_tile<kStrided>(smem + kOffdO + st * kStepBytes, tmdO, &bars->q_full[st], (wk.orders >> 12) & 15, 0,
                                    (s0 + s) * kStep, head, batch, bh);
            if (++st == kQStages) {
                st = 0;
                ph ^= 1;
            }
        }
        if (!ok) break;
        // all loads of this item are on their way: claim the next one now, and no earlier
        bars->ring.request();
        ++n_clc;
        ok = bars->ring.answer(w, &item, abort_flag, kWaitLimitCycles);
        if (!ok) break;
        ++w;
    }
    bars->asked_items = n_kv;
    bars->asked_steps = g;
    bars->asked_clc = n_clc;
}

// After a wait has run out: what is in flight lands before the CTA's shared memory goes away.  One thread, once every role has
// left: a stage's barrier counts the row terms of the edge warps too, and only then it is known which of them will not come.
template <bool kTerms>
__device__ __noinline__ void kv64_drain(Kv64Bars* bars) {
    int none = 0;
    const int n_clc = bars->asked_clc, n_kv = bars->asked_items, n_steps = bars->asked_steps;
    if (n_clc > 0) (void)mbar_wait(&bars->ring.answer_bar, (n_clc - 1) & 1, &none);
    for (int x = n_kv > 2 ? n_kv - 2 : 0; x < n_kv; ++x) (void)mbar_wait(&bars->kv_full[x & 1], (x >> 1) & 1, &none);
    for (int x = n_steps > kQStages ? n_steps - kQStages : 0; x < n_steps; ++x) {
        const int st = x % kQStages;
        if (!kTerms && *reinterpret_cast<volatile int*>(&bars->rows_of[st]) <= x) mbar_arrive(&bars->q_full[st]);
        (void)mbar_wait(&bars->q_full[st], (x / kQStages) & 1, &none);
    }
}

// Three UMMA issuers, each a whole warp in uniform control flow of which one elected lane issues.  Issuing takes as long as
// the products themselves (the queue in front of the tensor cores is short), so a single issuer leaves them idle whenever it
// waits: alone on an SM, a product of 172 clocks takes it 300 with one satisfied wait per product and 420 with three, while two
// issuers with three waits each keep the pipe full.  Beside the compute warps of its scheduler an issuer needs some 200
// clocks per wait: with one issuer a step of 64 queries took 1700 clocks, with two 1100, with three 800.  (dK and dP^T
// by one issuer, so that dP^T needs no wait for dK, were slower again, 980: what counts is the work per issuer.)

// acc[64 columns] = row terms + A B^T, A from TMEM and B K-major: 16 head-dim elements (8 columns, 32 bytes) per instruction
__device__ __forceinline__ void kv64_product(uint32_t t_acc, uint32_t t_a, uint32_t b, uint32_t ext_const, uint32_t ext) {
    constexpr uint32_t kIdescT = umma_idesc_bf16(128, kStep, 0, 0);
    const uint32_t hi = umma_desc_hi_sw128(1024), ext_hi = umma_desc_hi_plain(2 * kExtCore);
    umma_ss(t_acc, umma_desc_join(ext_const, ext_hi), umma_desc_join(ext, ext_hi), kIdescT, 0u);
#pragma unroll
    for (int k = 0; k < D / 16; ++k) umma_ts(t_acc, t_a + 8 * k, umma_desc_join(b + 2 * k, hi), kIdescT, 1u);
}

// S^T (kdP false): that of step g goes out as soon as the compute group has read that of step g - 2.
// dP^T (kdP true): as soon as dK of step g - 2 has read the dS^T that lies in the same columns.
template <bool kdP>
__device__ __forceinline__ void kv64_mma_sp(uint8_t* smem, Kv64Bars* bars, uint32_t tmem_base) {
    volatile int* abort_flag = &bars->abort_flag;
    const uint32_t b0 = umma_desc_lo(smem_u32(smem + (kdP ? kOffdO : kOffQ)), 16);
    const uint32_t ext0 = umma_desc_lo(smem_u32(smem + kOffExt), kExtCore);
    const uint32_t ext_const = ext0 + ((kQStages * kExtStep + (kdP ? kExtConst : 0)) >> 4);
    uint64_t* const full = kdP ? bars->dp_full : bars->s_full;
    uint64_t* const free = kdP ? bars->ds_done : bars->s_free;
    const bool el = elect_one();
    const int lane = threadIdx.x & 31;
    bool ok = true;
    int g = 0, st = 0;
    uint32_t ph = 0;
    for (int w = 0;; ++w) {
        const int n = bars->ring.take_steps(w, lane, abort_flag);
        if (n <= 0) {
            ok = (n == 0);
            break;
        }
        ok = mbar_wait(&bars->op_full[kdP], w & 1, abort_flag);
        if (!ok) break;
        for (int s = 0; s < n; ++s, ++g) {
            ok = mbar_wait(&bars->q_full[st], ph, abort_flag);
            if (ok) ok = mbar_wait(&free[g & 1], ((g >> 1) & 1) ^ 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            if (el) {
                kv64_product(tmem_base + (kdP ? kColdP : kColS) + kGroupCols * (g & 1), tmem_base + (kdP ? kColV : kColK),
                             b0 + st * (kStepBytes >> 4), ext_const, ext0 + st * (kExtStep >> 4));
                tc_commit(&full[g & 1]);
                if (s + 1 == n) tc_commit(&bars->op_free[kdP]);
            }
            __syncwarp();
            if (++st == kQStages) {
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

// dV and dK of each step, in order.
__device__ __forceinline__ void kv64_mma_acc(uint8_t* smem, Kv64Bars* bars, uint32_t tmem_base) {
    volatile int* abort_flag = &bars->abort_flag;
    constexpr uint32_t kIdescKV = umma_idesc_bf16(128, D, 0, 1);  // A from TMEM, B MN-major
    const uint32_t hi = umma_desc_hi_sw128(1024);
    const uint32_t q_m0 = umma_desc_lo(smem_u32(smem + kOffQ), kStepBytes);
    const uint32_t do_m0 = umma_desc_lo(smem_u32(smem + kOffdO), kStepBytes);
    const bool el = elect_one();
    const int lane = threadIdx.x & 31;
    bool ok = true;
    int g = 0, st = 0;
    for (int w = 0;; ++w) {
        const int n = bars->ring.take_steps(w, lane, abort_flag);
        if (n <= 0) {
            ok = (n == 0);
            break;
        }
        // the previous item's dV and dK must have been read out of TMEM before they are overwritten
        if (w > 0) ok = mbar_wait(&bars->dkv_free, (w - 1) & 1, abort_flag);
        if (!ok) break;
        for (int s = 0; s < n; ++s, ++g) {
            ok = mbar_wait(&bars->ready[g & 1], (g >> 1) & 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            if (el) {
                const uint32_t t_p = tmem_base + kColP + kGroupCols * (g & 1), t_ds = tmem_base + kColdP + kGroupCols * (g & 1);
                const uint32_t b_v = do_m0 + st * (kStepBytes >> 4), b_k = q_m0 + st * (kStepBytes >> 4);
#pragma unroll
                for (int k = 0; k < kStep / 16; ++k)  // 16 queries: 8 packed columns, 16 smem rows = 2048 bytes
                    umma_ts(tmem_base + kColdV, t_p + k * 8, umma_desc_join(b_v + k * 128, hi), kIdescKV,
                            (s > 0 || k > 0) ? 1u : 0u);
#pragma unroll
                for (int k = 0; k < kStep / 16; ++k)
                    umma_ts(tmem_base + kColdK, t_ds + k * 8, umma_desc_join(b_k + k * 128, hi), kIdescKV,
                            (s > 0 || k > 0) ? 1u : 0u);
                tc_commit(&bars->ds_done[g & 1]);
                tc_commit(&bars->q_empty[st]);
                if (s + 1 == n) tc_commit(&bars->dkv_full);
            }
            __syncwarp();
            if (++st == kQStages) st = 0;
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
template <bool kCausal>
__device__ __forceinline__ void kv64_compute(Kv64Bars* bars, uint32_t tmem_base, float scale, int grp, int cwarp, int lane) {
    volatile int* abort_flag = &bars->abort_flag;
    const uint32_t lane_base = 32u * cwarp;
    const int r = lane_base + lane;  // local key row
    const float c = fmaxf(scale, kLeastScale) * kLog2e;
    const uint64_t c2 = f32x2_pack(c, c);
    const uint32_t t_s = tmem_addr(tmem_base, lane_base, kColS + kGroupCols * grp);
    const uint32_t t_dp = t_s + (kColdP - kColS), t_p = t_s + (kColP - kColS);
    bool ok = true;
    int g = 0;         // steps of all items so far
    uint32_t ph = 0;   // phase of this group's barriers

    for (int w = 0;; ++w) {
        const int n = bars->ring.take_steps(w, lane, abort_flag);
        if (n <= 0) {
            ok = (n == 0);
            break;
        }
        for (int s = (g ^ grp) & 1; s < n; s += 2, ph ^= 1) {
            ok = mbar_wait(&bars->s_full[grp], ph, abort_flag);
            if (!ok) break;
            tc_fence_after();
            uint32_t pf[kStep];
            tmem_ld_x32(t_s, pf);
            tmem_ld_x32(t_s + 32, pf + 32);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->s_free[grp]);
            // the scores become fp32 probabilities in place
#pragma unroll
            for (int i = 0; i < kStep; i += 2) {
                float x0, x1;
                f32x2_unpack(f32x2_mul(f32x2_pack(__uint_as_float(pf[i]), __uint_as_float(pf[i + 1])), c2), x0, x1);
                pf[i] = __float_as_uint(ex2_approx(x0));
                pf[i + 1] = __float_as_uint(ex2_approx(x1));
            }
            // Keep key <= query (the first steps of a causal item).  Keys past the end of the sequence need no mask: their
            // rows are not stored.
            const int first = r - s * kStep;  // first kept query of the step
            if (kCausal && s < kBlockK / kStep) {
#pragma unroll
                for (int i = 0; i < kStep; ++i)
                    if (i < first) pf[i] = 0u;
            }
            // dP^T of this step was issued after dV of the group's previous one had read the P^T columns
            ok = mbar_wait(&bars->dp_full[grp], ph, abort_flag);
            if (!ok) break;
            tc_fence_after();
            uint32_t dv[16];
            tmem_ld_x16(t_dp, dv);
#pragma unroll
            for (int x = 0; x < kStep; x += 32) {
                uint32_t pk[16];
#pragma unroll
                for (int y = 0; y < 16; ++y)
                    pk[y] = pack_bf16x2(__uint_as_float(pf[x + 2 * y]), __uint_as_float(pf[x + 2 * y + 1]));
                tmem_st_x16(t_p + x / 2, pk);
            }
            // dS^T from the unrounded P^T: only what feeds a contraction is rounded (paper Section 4.3); 16 queries at a
            // time, over dP^T columns that have been read
#pragma unroll
            for (int x = 0; x < kStep; x += 16) {
                tmem_wait_ld();
                uint32_t dd[8];
#pragma unroll
                for (int y = 0; y < 8; ++y) {
                    float d0, d1;
                    f32x2_unpack(f32x2_mul(f32x2_pack(__uint_as_float(pf[x + 2 * y]), __uint_as_float(pf[x + 2 * y + 1])),
                                           f32x2_pack(__uint_as_float(dv[2 * y]), __uint_as_float(dv[2 * y + 1]))), d0, d1);
                    dd[y] = pack_bf16x2(d0, d1);
                }
                if (x + 16 < kStep) tmem_ld_x16(t_dp + x + 16, dv);
                tmem_st_x8(t_dp + x / 2, dd);
            }
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->ready[grp]);
        }
        if (!ok) break;
        g += n;
    }
}

// Edge warps (warp `ow` of four, thread = key row): what happens at the ends of an item and on the way into a step.
//   K and V of an item from shared into tensor memory, each as soon as the last product that reads these columns is done;
//   the row terms of every step into its stage, the steps dealt out among the four warps, two queries per lane;
//   dV and dK * scale of a finished item as bf16 into shared memory and out with TMA stores.
// The stages of an item's first kQStages steps are handed back by the item before, whose dV and dK may wait till then; the
// later ones only after dV and dK have been read out.
template <bool kStrided, bool kTerms>
__device__ __forceinline__ void kv64_edges(uint8_t* smem, Kv64Bars* bars, uint32_t tmem_base, const CUtensorMap* tmdK,
                                           const CUtensorMap* tmdV, const float* __restrict__ LSE,
                                           const float* __restrict__ Delta, float scale, const Kv64Work& wk, int ow, int lane) {
    volatile int* abort_flag = &bars->abort_flag;
    const uint32_t lane_base = 32u * ow;
    const int r = lane_base + lane;
    const bool leader = (ow == 0 && lane == 0);
    const float inv_scale = 1.0f / fmaxf(scale, kLeastScale);
    bool ok = true;

    // K (v = 0) or V (v = 1) of the w-th item: a row of 64 bf16 numbers is 32 columns
    auto operand = [&](int w, int v) -> bool {
        const int ks = w & 1;
        if (v == 0 && !mbar_wait(&bars->kv_full[ks], (w >> 1) & 1, abort_flag)) return false;
        uint32_t a[32];
#pragma unroll
        for (int ch = 0; ch < 8; ++ch) {
            const uint4 x = *reinterpret_cast<const uint4*>(smem + (v ? kOffV : kOffK) + ks * kTileBytes + r * 128 +
                                                            ((ch ^ (r & 7)) << 4));
            a[4 * ch] = x.x, a[4 * ch + 1] = x.y, a[4 * ch + 2] = x.z, a[4 * ch + 3] = x.w;
        }
        if (w > 0 && !mbar_wait(&bars->op_free[v], (w - 1) & 1, abort_flag)) return false;
        tc_fence_after();
        __syncwarp();
        tmem_st_x32(tmem_addr(tmem_base, lane_base, v ? kColV : kColK), a);
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
            if (v == 1) mbar_arrive(&bars->kv_empty[ks]);
            mbar_arrive(&bars->op_full[v]);
        }
        return true;
    };
    // Row terms of the item's steps in [from, to) that are this warp's; g0: steps of all items before this one.
    auto rows = [&](int bh, int s0, int g0, int from, int to) -> bool {
        const size_t base = static_cast<size_t>(bh) * wk.T;
        uint8_t* const row = smem + kOffExt + (lane >> 3) * 2 * kExtCore + (lane & 7) * 16;
        constexpr int kNext32 = 32 / 8 * 2 * kExtCore;  // the row 32 queries on
        for (int s = from + ((ow - g0 - from) & 3); s < to; s += 4) {
            const int g = g0 + s, st = g % kQStages;
            RowTerms t[2];
#pragma unroll
            for (int x = 0; x < 2; ++x) {  // (past L1: there was no griddep_wait)
                const int q = (s0 + s) * kStep + lane + 32 * x;
                t[x] = row_terms((q < wk.T) ? -__ldcg(LSE + base + q) * inv_scale : -kMostLse,
                                 (q < wk.T) ? -__ldcg(Delta + base + q) : 0.f);
            }
            const bool any_odd = __any_sync(0xffffffffu, t[0].odd || t[1].odd);
            if (!mbar_wait(&bars->q_empty[st], ((g / kQStages) & 1) ^ 1, abort_flag)) return false;
#pragma unroll
            for (int x = 0; x < 2; ++x) *reinterpret_cast<uint4*>(row + st * kExtStep + x * kNext32) = t[x].first;
            // (a stage is written by two of the warps in turn: the flag says what the one before left behind)
            if (any_odd || *reinterpret_cast<volatile int*>(&bars->odd_rows[st]) != 0) {
#pragma unroll
                for (int x = 0; x < 2; ++x)
                    *reinterpret_cast<uint4*>(row + st * kExtStep + x * kNext32 + kExtCore) = t[x].second;
                __syncwarp();
                if (lane == 0) *reinterpret_cast<volatile int*>(&bars->odd_rows[st]) = any_odd;
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                *reinterpret_cast<volatile int*>(&bars->rows_of[st]) = g + 1;
                mbar_arrive(&bars->q_full[st]);
            }
        }
        return true;
    };
    // dV and dK of the w-th item
    auto write_out = [&](int w, int kt, int bh) -> bool {
        if (!mbar_wait(&bars->dkv_full, w & 1, abort_flag)) return false;
        tc_fence_after();
        __syncwarp();
        uint32_t pk[2][32];
#pragma unroll
        for (int which = 0; which < 2; ++which) {
            const uint32_t t_o = tmem_addr(tmem_base, lane_base, which ? kColdK : kColdV);
            const float f = which ? scale : 1.0f;
#pragma unroll
            for (int cb = 0; cb < D; cb += 32) {
                uint32_t a[32];
                tmem_ld_x32(t_o + cb, a);
                tmem_wait_ld();
#pragma unroll
                for (int x = 0; x < 16; ++x)
                    pk[which][cb / 2 + x] = pack_bf16x2(__uint_as_float(a[2 * x]) * f, __uint_as_float(a[2 * x + 1]) * f);
            }
        }
        tc_fence_before();
        if (leader) {  // the buffers are free once what was sent from them last has been read
            bulk_wait_group_read<0>();
            mbar_arrive(&bars->stage_free);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->dkv_free);
        if (!mbar_wait(&bars->stage_free, w & 1, abort_flag)) return false;
#pragma unroll
        for (int which = 0; which < 2; ++which)
#pragma unroll
            for (int x = 0; x < 8; ++x)
                *reinterpret_cast<uint4*>(smem + kOffOut + which * kTileBytes + r * 128 + ((x ^ (r & 7)) << 4)) =
                    make_uint4(pk[which][4 * x], pk[which][4 * x + 1], pk[which][4 * x + 2], pk[which][4 * x + 3]);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->staged);
        bool leader_ok = true;
        if (leader) {
            leader_ok = mbar_wait(&bars->staged, w & 1, abort_flag);
            if (leader_ok) {
                const int hh = kStrided ? bh % wk.H : 0, bb = kStrided ? bh / wk.H : 0;
                tma_store_tile<kStrided>(tmdV, smem + kOffOut, (wk.orders >> 20) & 15, 0, kt * kBlockK, hh, bb, bh);
                tma_store_tile<kStrided>(tmdK, smem + kOffOut + kTileBytes, (wk.orders >> 16) & 15, 0, kt * kBlockK, hh, bb, bh);
                bulk_commit_group();
            }
        }
        return __all_sync(0xffffffffu, leader_ok);
    };

    int g0 = 0, kt_out = 0, bh_out = 0;
    for (int w = 0; ok; ++w) {
        int item = 0;
        const int taken = bars->ring.take_steps(w, lane, abort_flag, &item);
        if (taken <= 0) {
            if (taken == 0 && w > 0) (void)write_out(w - 1, kt_out, bh_out);
            break;
        }
        int kt, bh, s0, n;
        wk.get(item, &kt, &bh, &s0, &n);
        if (!kTerms) ok = rows(bh, s0, g0, 0, min(n, 2));
        if (ok) ok = operand(w, 0);
        if (ok) ok = operand(w, 1);
        if (ok && !kTerms) ok = rows(bh, s0, g0, 2, min(n, kQStages));
        if (ok && w > 0) ok = write_out(w - 1, kt_out, bh_out);
        if (ok && !kTerms) ok = rows(bh, s0, g0, kQStages, n);
        kt_out = kt;
        bh_out = bh;
        g0 += n;
    }
    if (leader) bulk_wait_group<0>();  // dV and dK must be complete before the kernel ends
}

template <bool kCausal, bool kStrided, bool kTerms>
__global__ void __launch_bounds__(kThreads, 1)
attn_dkdv64_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                   const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmdO,
                   const __grid_constant__ CUtensorMap tmdK, const __grid_constant__ CUtensorMap tmdV,
                   const float* __restrict__ LSE, const float* __restrict__ Delta, const uint8_t* __restrict__ terms, int T, int BH,
                   int H, uint32_t orders, float scale, int* __restrict__ dev_status) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    Kv64Bars* bars = reinterpret_cast<Kv64Bars*>(smem + kOffBar);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const Kv64Work wk{BH, T, H, orders, kCausal};

    // The kernel before this one in the stream is the dQ kernel, of which nothing is needed: it need not have completed (ptx.cuh).
    // The threads that will read global memory, the producer and the edge warps, see to it while the others set up.
    if (threadIdx.x == 0 || (!kTerms && warp >= 12)) griddep_taken_over();
    if (threadIdx.x == 64) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(&bars->kv_full[s], 1);
            mbar_init(&bars->kv_empty[s], 4);
            mbar_init(&bars->s_full[s], 1);
            mbar_init(&bars->s_free[s], 4);
            mbar_init(&bars->dp_full[s], 1);
            mbar_init(&bars->ready[s], 4);
            mbar_init(&bars->ds_done[s], 1);
            mbar_init(&bars->op_full[s], 4);
            mbar_init(&bars->op_free[s], 1);
        }
        for (int s = 0; s < kQStages; ++s) {
            mbar_init(&bars->q_full[s], kTerms ? 1 : 2);  // the producer, and the edge warp that writes the row terms
            mbar_init(&bars->q_empty[s], 1);
            bars->odd_rows[s] = 0;
            bars->rows_of[s] = 0;
        }
        mbar_init(&bars->dkv_full, 1);
        mbar_init(&bars->dkv_free, 4);
        mbar_init(&bars->staged, 4);
        mbar_init(&bars->stage_free, 1);
        for (int s = 0; s < 3; ++s) mbar_init(&bars->drain[s], 1);
        bars->ring.init(kWorkConsumers);
        bars->abort_flag = 0;
        fence_mbar_init();
        tma_prefetch_desc(&tmQ);
        tma_prefetch_desc(&tmK);
        tma_prefetch_desc(&tmV);
        tma_prefetch_desc(&tmdO);
        tma_prefetch_desc(&tmdK);
        tma_prefetch_desc(&tmdV);
    }
    // zeros in the stages of the row terms, then the constants
    for (int i = threadIdx.x; i < kExtBytes / 16; i += kThreads) {
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        const bool first_half = ((i >> 3) & 1) == 0;  // core matrix of columns 0-7
        const int k = i - kQStages * kExtStep / 16;
        if (k >= 0 && k < kExtConst / 16 && first_half) v = make_uint4(0x00003f80u, 0x00003f80u, 0x00003f80u, 0u);
        if (k >= kExtConst / 16 && first_half) v = make_uint4(0x3f800000u, 0x3f800000u, 0x3f800000u, 0u);
        if (k >= kExtConst / 16 && !first_half) v.x = __bfloat16_as_ushort(__float2bfloat16_rn(kMostLse));
        *reinterpret_cast<uint4*>(smem + kOffExt + 16 * i) = v;
    }
    fence_proxy_async_smem();
    if (warp == 1) {
        tmem_alloc(&bars->tmem_base, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = bars->tmem_base;
    griddep_launch_dependents();

    if (warp == 0) {
        if (lane == 0) kv64_producer<kStrided, kTerms>(&tmQ, &tmK, &tmV, &tmdO, terms, smem, bars, wk);
    } else if (warp == 1) {
        kv64_mma_sp<false>(smem, bars, tmem_base);
    } else if (warp == 2) {
        kv64_mma_sp<true>(smem, bars, tmem_base);
    } else if (warp == 3) {
        kv64_mma_acc(smem, bars, tmem_base);
    } else if (warp >= 12) {
        kv64_edges<kStrided, kTerms>(smem, bars, tmem_base, &tmdK, &tmdV, LSE, Delta, scale, wk, warp & 3, lane);
    } else {
        kv64_compute<kCausal>(bars, tmem_base, scale, (warp - 4) >> 2, warp & 3, lane);
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, kTmemCols);
    if (threadIdx.x == 0 && bars->abort_flag != 0) kv64_drain<kTerms>(bars);
    griddep_wait();  // what waits for this kernel waits for dQ too
    if (threadIdx.x == 0 && bars->abort_flag != 0) atomicExch(dev_status, kDevTimeout);
}

}  // namespace

cudaError_t configure_attn_dkdv64() {
    auto set = [](auto kernel) {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    };
    cudaError_t e = set(attn_dkdv64_kernel<true, false, false>);
    if (e == cudaSuccess) e = set(attn_dkdv64_kernel<false, false, false>);
    if (e == cudaSuccess) e = set(attn_dkdv64_kernel<true, false, true>);
    if (e == cudaSuccess) e = set(attn_dkdv64_kernel<true, true, true>);
    if (e == cudaSuccess) e = set(attn_dkdv64_kernel<false, false, true>);
    if (e == cudaSuccess) e = set(attn_dkdv64_kernel<false, true, true>);
    return e;
}

cudaError_t launch_row_terms64(const float* LSE, const float* Delta, void* terms, const AttnShape& s, cudaStream_t stream) {
    const int n_steps = (s.T + kStep - 1) / kStep;
    const long long rows = static_cast<long long>(s.B) * s.H * n_steps * kStep;
    return launch_overlapped(row_terms64_kernel, dim3(static_cast<unsigned>((rows + 255) / 256)), dim3(256), 0, stream, LSE, Delta,
                             static_cast<uint8_t*>(terms), s.T, n_steps, rows, 1.0f / fmaxf(s.scale, kLeastScale));
}

cudaError_t launch_attn_dkdv64(const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV,
                               const CUtensorMap& tmdO, const CUtensorMap& tmdK, const CUtensorMap& tmdV, bool strided,
                               uint32_t orders, const float* LSE, const float* Delta, const void* terms, const AttnShape& s,
                               int* dev_status, cudaStream_t stream) {
    if (strided && terms == nullptr) return cudaErrorNotSupported;  // (only the deterministic entry point has no workspace)
    const int n_tiles = (s.T + kBlockK - 1) / kBlockK, BH = s.B * s.H;
    const dim3 grid(static_cast<unsigned>(n_tiles) * BH);  // one CTA per item; those that do not start are taken over
    auto go = [&](auto kernel) {
        return launch_overlapped(kernel, grid, dim3(kThreads), kSmemBytes, stream, tmQ, tmK, tmV, tmdO, tmdK, tmdV, LSE, Delta,
                                 static_cast<const uint8_t*>(terms), s.T, BH, s.H, orders, s.scale, dev_status);
    };
    if (terms == nullptr) return s.causal ? go(attn_dkdv64_kernel<true, false, false>) : go(attn_dkdv64_kernel<false, false, false>);
    if (s.causal) return strided ? go(attn_dkdv64_kernel<true, true, true>) : go(attn_dkdv64_kernel<true, false, true>);
    return strided ? go(attn_dkdv64_kernel<false, true, true>) : go(attn_dkdv64_kernel<false, false, true>);
}

}  // namespace nova
