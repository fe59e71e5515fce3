// dK and dV of the two-kernel backward at D = 128 (paper Section 4.2, "The Backward Pass": one kernel reduces dQ over
// keys, the other reduces dK and dV over queries; the probability matrix is rebuilt from the saved log-sum-exp, never
// stored; the causal loop bound is raised so that queries above the diagonal are never visited).
//
// A work item is one 128-key tile of one head; its queries go by in steps of 64.  As in the fused kernel everything is
// transposed, keys on the lanes of tensor memory, so that P^T and dS^T feed the tensor cores from where they are made:
//   S^T  = K_j Q_s^T,  dP^T = V_j dO_s^T                       (smem x smem -> one of two buffers in TMEM)
//   P^T  = exp2(S^T*c - LSE*log2e),  dS^T = P^T * (dP^T - Delta)   (bf16, over the S^T and dP^T they came from)
//   dV  += P^T dO_s,  dK += dS^T Q_s                           (TMEM x smem, dO and Q read MN-major)
// Items are handed out dynamically (WorkRing), heaviest first within a chunk of heads whose tensors stay in L2
// together.  512 threads:
//   warp 0      TMA producer: K_j double-buffered, V_j, and Q_s and dO_s through a ring of 64-query stages
//   warp 1      UMMA issuer: S^T and dP^T run two steps ahead of dV and dK, across item boundaries
//   warp 2      row loader: -LSE*log2e and -Delta of a step into shared memory
//   warps 4-7   compute group 0, warps 8-11 group 1: the steps alternate between the groups; a thread has one key
//               row and the 64 queries of its step
//   warps 12-15 send dV and dK of a finished item out, through the item's own K buffer, which nothing reads any more,
//               while the compute warps are in the next item
#include "kernels.h"
#include "ptx.cuh"

namespace nova {
namespace {

constexpr int D = 128;
constexpr int kThreads = 512;
constexpr int kTmemCols = 512;
constexpr int kStep = kKeyStep;              // queries per step
constexpr int kHalfStepBytes = kStep * 128;  // one [64 rows x 64 bf16] box
constexpr int kHalves = D / kBoxCols;
constexpr int kTileBytes = kHalves * kHalfTileBytes;
constexpr int kStepBytes = kHalves * kHalfStepBytes;
constexpr int kQStages = 4;
constexpr int kBufs = 2;                     // buffers of S^T and dP^T, one per compute group
constexpr int kRowStages = 4;
constexpr int kWorkConsumers = 2 + 8 + 4;    // issuer, row loader, compute warps, write-out warps
static_assert(kQStages >= kBufs, "the issuer runs kBufs steps ahead");

// One V buffer and four stages of Q and dO rather than two and three: with three the loads of a step (32 KB, 1300 clocks
// from L2 with every SM loading) came too late for it, while V of the next item has the last two steps of this one.
constexpr int kOffK = 0;                                 // [2]
constexpr int kOffV = 2 * kTileBytes;
constexpr int kOffQ = 3 * kTileBytes;                    // [kQStages]
constexpr int kOffdO = kOffQ + kQStages * kStepBytes;    // [kQStages]
constexpr int kOffRow = kOffdO + kQStages * kStepBytes;  // [kRowStages] x (-LSE*log2e[64], -Delta[64])
constexpr int kOffBar = kOffRow + kRowStages * 2 * kStep * 4;
// There is no room to realign the window: the kernel checks that it starts on a 1024-byte boundary.
constexpr int kSmemBytes = kOffBar + 512;
static_assert(kSmemBytes <= 232448, "exceeds the shared memory of one CTA");
constexpr int kColdV = 0, kColdK = D, kColBuf = 2 * D;   // + 128 * buffer: S^T / P^T, then dP^T / dS^T

struct KvBars {
    uint64_t k_full[2], k_empty[2], v_full, v_empty;
    uint64_t q_full[kQStages], q_empty[kQStages];
    uint64_t row_full[kRowStages], row_empty[kRowStages];
    uint64_t sp_full[kBufs], ready[kBufs];  // per buffer: UMMA -> compute group, compute group -> UMMA
    uint64_t dkv_full, dkv_free;            // dV and dK of an item complete; read out of TMEM
    uint64_t staged, stage_free;            // the write-out warps among themselves
    uint64_t drain;
    WorkRing ring;
    uint32_t tmem_base;
    int abort_flag;
};
static_assert(sizeof(KvBars) <= 512, "barrier block");

// Work items: 128-key tiles; heads in chunks, heaviest tiles first within a chunk.
struct KvWork {
    int BH, n_tiles, chunk, T, H;
    uint32_t orders;  // coordinate orders of the Q, K, V, dO, dK, dV tensor maps, four bits each
    bool causal;
    // Key tile, head, first step and number of steps of item `idx`.
    __device__ __forceinline__ void get(int idx, int* kt, int* bh, int* s0, int* n) const {
        const int per_chunk = chunk * n_tiles;
        const int ck = idx / per_chunk, in = idx - ck * per_chunk;
        const int heads = min(chunk, BH - ck * chunk);
        *kt = in / heads;
        *bh = ck * chunk + in - *kt * heads;
        *s0 = causal ? *kt * (kBlockK / kStep) : 0;
        *n = (T + kStep - 1) / kStep - *s0;
    }
};

template <bool kStrided>
__device__ __forceinline__ void kv_producer(const CUtensorMap* tmQ, const CUtensorMap* tmK, const CUtensorMap* tmV,
                                            const CUtensorMap* tmdO, uint8_t* smem, KvBars* bars, const KvWork& wk) {
    volatile int* abort_flag = &bars->abort_flag;
    int armed_k[2] = {-1, -1}, armed_v = -1, armed_q[kQStages];
    for (int s = 0; s < kQStages; ++s) armed_q[s] = -1;
    bool ok = true, clc_pending = false;
    int w = 0, st = 0;
    uint32_t ph = 0;
    int item = blockIdx.x;
    for (;;) {
        ok = bars->ring.publish(w, item, abort_flag, kWaitLimitCycles);
        if (!ok || item < 0) break;
        int kt, bh, s0, n;
        wk.get(item, &kt, &bh, &s0, &n);
        const int head = kStrided ? bh % wk.H : 0, batch = kStrided ? bh / wk.H : 0;
        const int ks = w & 1;
        ok = mbar_wait(&bars->k_empty[ks], ((w >> 1) & 1) ^ 1, abort_flag);
        if (!ok) break;
        mbar_expect_tx(&bars->k_full[ks], kTileBytes);  // rows past T arrive as zeros
        armed_k[ks] = (w >> 1) & 1;
#pragma unroll
        for (int h = 0; h < kHalves; ++h)
            tma_load_tile<kStrided>(smem + kOffK + ks * kTileBytes + h * kHalfTileBytes, tmK, &bars->k_full[ks],
                                    (wk.orders >> 4) & 15, h * kBoxCols, kt * kBlockK, head, batch, bh);
        for (int s = 0; s < n; ++s) {
            ok = mbar_wait(&bars->q_empty[st], ph ^ 1, abort_flag);
            if (!ok) break;
            mbar_expect_tx(&bars->q_full[st], 2 * kStepBytes);
            armed_q[st] = ph;
#pragma unroll
            for (int h = 0; h < kHalves; ++h) {
                tma_load_tile<kStrided>(smem + kOffQ + st * kStepBytes + h * kHalfStepBytes, tmQ, &bars->q_full[st],
                                        wk.orders & 15, h * kBoxCols, (s0 + s) * kStep, head, batch, bh);
                tma_load_tile<kStrided>(smem + kOffdO + st * kStepBytes + h * kHalfStepBytes, tmdO, &bars->q_full[st],
                                        (wk.orders >> 12) & 15, h * kBoxCols, (s0 + s) * kStep, head, batch, bh);
            }
            if (++st == kQStages) {
                st = 0;
                ph ^= 1;
            }
            if (s == 0) {  // V after the first queries: its buffer is the last thing the previous item hands back
                ok = mbar_wait(&bars->v_empty, (w & 1) ^ 1, abort_flag);
                if (!ok) break;
                mbar_expect_tx(&bars->v_full, kTileBytes);
                armed_v = w & 1;
#pragma unroll
                for (int h = 0; h < kHalves; ++h)
                    tma_load_tile<kStrided>(smem + kOffV + h * kHalfTileBytes, tmV, &bars->v_full, (wk.orders >> 8) & 15,
                                            h * kBoxCols, kt * kBlockK, head, batch, bh);
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
        for (int s = 0; s < 2; ++s)
            if (armed_k[s] >= 0) (void)mbar_wait(&bars->k_full[s], armed_k[s], &none);
        if (armed_v >= 0) (void)mbar_wait(&bars->v_full, armed_v, &none);
        for (int s = 0; s < kQStages; ++s)
            if (armed_q[s] >= 0) (void)mbar_wait(&bars->q_full[s], armed_q[s], &none);
    }
}

// UMMA issuer: the whole warp in uniform control flow, one elected lane issues.
__device__ __forceinline__ void kv_mma(uint8_t* smem, KvBars* bars, uint32_t tmem_base, const KvWork& wk) {
    volatile int* abort_flag = &bars->abort_flag;
    constexpr uint32_t kIdescT = umma_idesc_bf16(128, kStep, 0, 0);  // S^T, dP^T
    constexpr uint32_t kIdescKV = umma_idesc_bf16(128, D, 0, 1);     // dV, dK: A from TMEM, B MN-major
    const uint32_t hi = umma_desc_hi_sw128(1024);
    const uint32_t k_k0 = umma_desc_lo(smem_u32(smem + kOffK), 16), v_k0 = umma_desc_lo(smem_u32(smem + kOffV), 16);
    const uint32_t q_k0 = umma_desc_lo(smem_u32(smem + kOffQ), 16), do_k0 = umma_desc_lo(smem_u32(smem + kOffdO), 16);
    const uint32_t q_m0 = umma_desc_lo(smem_u32(smem + kOffQ), kHalfStepBytes);
    const uint32_t do_m0 = umma_desc_lo(smem_u32(smem + kOffdO), kHalfStepBytes);
    const bool el = elect_one();
    const int lane = threadIdx.x & 31;
    bool ok = true;

    // acc[64 columns] = A B^T, both K-major, 16 head-dim elements (32 bytes) per instruction
    auto product = [&](uint32_t t_acc, uint32_t a, uint32_t b) {
#pragma unroll
        for (int k = 0; k < D / 16; ++k)
            umma_ss(t_acc, umma_desc_join(a + (((k / 4) * kHalfTileBytes + (k % 4) * 32) >> 4), hi),
                    umma_desc_join(b + (((k / 4) * kHalfStepBytes + (k % 4) * 32) >> 4), hi), kIdescT, k > 0 ? 1u : 0u);
    };

    // Two cursors over the same sequence of steps: `a` is where S^T and dP^T go next, `c` where dV and dK do.  The first
    // may be in a later item.  Within an item its loads may be waited for: a stage that a step needs was handed back at
    // least kQStages steps before, i.e. by what `c` has already done.  For the next item's first step nothing is waited
    // for while there are steps between the cursors (its loads may depend on stages that only `c` frees).
    int w_a = 0, left_a = 0;          // items taken by `a`; steps left in the latest
    bool kv_seen = true, more = true; // its K and V have landed; there may be further items
    int st_a = 0, buf_a = 0;          // Q stage and buffer of `a`
    uint32_t ph_a = 0;
    int n_of[2] = {0, 0};             // steps of item w, by w & 1, for `c`
    int w_c = 0, done_c = 0;          // item of `c` and its steps so far
    int st_c = 0, buf_c = 0;
    uint32_t rdy_ph = 0;              // phase of ready[buf_c]
    int ahead = 0;                    // steps between the cursors

    // Are K, V, Q and dO of the next step of `a` there?  False without an error: not yet, or no items left.
    auto probe = [&]() -> bool {
        if (!more) return false;
        if (left_a > 0 && kv_seen) {
            ok = mbar_wait(&bars->q_full[st_a], ph_a, abort_flag);
            return ok;
        }
        const bool block = ahead == 0;
        if (left_a == 0) {
            if (w_a - w_c >= 2) return false;  // the number of steps of the item of `c` would be overwritten
            if (!block && !bars->ring.published(w_a)) return false;
            const int item = bars->ring.take(w_a, lane, abort_flag, kWaitLimitCycles);
            if (item < 0) {
                ok = (item == -1);
                more = false;
                return false;
            }
            int kt, bh, s0, n;
            wk.get(item, &kt, &bh, &s0, &n);
            left_a = n;
            if (w_a & 1) n_of[1] = n;
            else n_of[0] = n;
            ++w_a;
            kv_seen = false;
        }
        const uint32_t p = ((w_a - 1) >> 1) & 1;
        if (block) {
            ok = mbar_wait(&bars->k_full[(w_a - 1) & 1], p, abort_flag);
            if (ok) ok = mbar_wait(&bars->v_full, (w_a - 1) & 1, abort_flag);
            if (ok) ok = mbar_wait(&bars->q_full[st_a], ph_a, abort_flag);
            kv_seen = ok;
        } else {
            const bool there = mbar_test(&bars->k_full[(w_a - 1) & 1], p) && mbar_test(&bars->v_full, (w_a - 1) & 1) &&
                               mbar_test(&bars->q_full[st_a], ph_a);
            kv_seen = __all_sync(0xffffffffu, there);
        }
        return kv_seen;
    };
    // S^T and dP^T of the next step of `a`.  The buffer is free: the dV and dK products that read its P^T and dS^T were
    // queued before this point.
    auto issue_sp = [&]() {
        tc_fence_after();
        if (el) {
            const int ks = (w_a - 1) & 1;
            const uint32_t t_b = tmem_base + kColBuf + 128 * buf_a;
            product(t_b, k_k0 + ks * (kTileBytes >> 4), q_k0 + st_a * (kStepBytes >> 4));
            product(t_b + 64, v_k0, do_k0 + st_a * (kStepBytes >> 4));
            tc_commit(&bars->sp_full[buf_a]);
            if (left_a == 1) tc_commit(&bars->v_empty);  // the item's last step
        }
        __syncwarp();
        --left_a;
        ++ahead;
        if (++st_a == kQStages) {
            st_a = 0;
            ph_a ^= 1;
        }
        buf_a ^= 1;
    };

    for (;;) {
        while (ahead < kBufs && probe()) issue_sp();
        if (!ok || ahead == 0) break;  // given up, or no items left
        // The loads of the step that takes over the buffer of the oldest one are looked for before that one is waited
        // for: nothing then stands between its dV and dK and the next S^T and dP^T (worth 20 %: the tensor pipe idles
        // while its issuer waits).
        const bool next_there = ahead == kBufs && probe();
        if (!ok) break;
        // ---- dV and dK of the oldest step
        ok = mbar_wait(&bars->ready[buf_c], rdy_ph, abort_flag);
        // the previous item's dV and dK must have been read out of TMEM before they are overwritten
        if (ok && done_c == 0 && w_c > 0) ok = mbar_wait(&bars->dkv_free, (w_c - 1) & 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const bool last = done_c + 1 == ((w_c & 1) ? n_of[1] : n_of[0]);
        if (el) {
            const uint32_t t_b = tmem_base + kColBuf + 128 * buf_c;
            const uint32_t b_v = do_m0 + st_c * (kStepBytes >> 4), b_k = q_m0 + st_c * (kStepBytes >> 4);
#pragma unroll
            for (int k = 0; k < kStep / 16; ++k)  // 16 queries: 8 packed columns, 16 smem rows = 2048 bytes
                umma_ts(tmem_base + kColdV, t_b + k * 8, umma_desc_join(b_v + k * 128, hi), kIdescKV,
                        (done_c > 0 || k > 0) ? 1u : 0u);
#pragma unroll
            for (int k = 0; k < kStep / 16; ++k)
                umma_ts(tmem_base + kColdK, t_b + 64 + k * 8, umma_desc_join(b_k + k * 128, hi), kIdescKV,
                        (done_c > 0 || k > 0) ? 1u : 0u);
            tc_commit(&bars->q_empty[st_c]);
            if (last) tc_commit(&bars->dkv_full);
        }
        __syncwarp();
        if (next_there) issue_sp();
        --ahead;
        if (++st_c == kQStages) st_c = 0;
        rdy_ph ^= buf_c;  // after the second buffer
        buf_c ^= 1;
        if (last) {
            done_c = 0;
            ++w_c;
        } else {
            ++done_c;
        }
    }
    if (!ok) {
        int none = 0;
        if (el) tc_commit(&bars->drain);
        __syncwarp();
        (void)mbar_wait(&bars->drain, 0, &none);
    }
}

// Row loader (one warp): -LSE*log2e and -Delta of each step, negated so that the compute warps fold them in with a packed
// fma / add.  Queries past the end of the sequence get -inf, so that their P is exactly 0.  A NaN (or + inf) becomes 3e38:
// P of that query is infinite where it is kept, as unusable as NaN, but 0 where the causal mask puts -inf in front of the
// sum, so that it reaches no key behind it.  (Making what is masked zero in the compute warps, per packed word or in a
// branch that is not taken, cost 0.8 to 1.5 % of the training pass at B=4, H=32, T=1000.)  The loads of four steps are in
// flight together.
__device__ __forceinline__ void kv_row_loader(KvBars* bars, float* row_buf, const float* __restrict__ LSE,
                                              const float* __restrict__ Delta, const KvWork& wk, int lane) {
    volatile int* abort_flag = &bars->abort_flag;
    constexpr int kDeep = 4;
    int g = 0;
    for (int w = 0;; ++w) {
        const int item = bars->ring.take(w, lane, abort_flag, kWaitLimitCycles);
        if (item < 0) return;
        int kt, bh, s0, n;
        wk.get(item, &kt, &bh, &s0, &n);
        const size_t base = static_cast<size_t>(bh) * wk.T;
        for (int s = 0; s < n; s += kDeep) {
            float l[kDeep][2], d[kDeep][2];
#pragma unroll
            for (int u = 0; u < kDeep; ++u)
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    const int q = (s0 + s + u) * kStep + lane + 32 * x;
                    l[u][x] = (q < wk.T) ? LSE[base + q] : INFINITY;
                    d[u][x] = (q < wk.T) ? Delta[base + q] : 0.f;
                }
#pragma unroll
            for (int u = 0; u < kDeep; ++u) {
                if (s + u >= n) break;
                const int b = g % kRowStages;
                if (!mbar_wait(&bars->row_empty[b], ((g / kRowStages) & 1) ^ 1, abort_flag)) return;
                float* r = row_buf + b * 2 * kStep;
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    const float nl = -l[u][x] * kLog2e;
                    r[lane + 32 * x] = nl < 3e38f ? nl : 3e38f;
                    r[kStep + lane + 32 * x] = -d[u][x];
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars->row_full[b]);
                ++g;
            }
        }
    }
}

// Compute group `grp` (steps g with g % 2 == grp, which are those of buffer `grp`), warp `cwarp` of it.
template <bool kCausal>
__device__ __forceinline__ void kv_compute(const uint8_t* smem, KvBars* bars, uint32_t tmem_base, float scale,
                                           const KvWork& wk, int grp, int cwarp, int lane) {
    volatile int* abort_flag = &bars->abort_flag;
    const uint32_t lane_base = 32u * cwarp;
    const int r = lane_base + lane;  // local key row
    const float c = scale * kLog2e;
    const uint64_t c2 = f32x2_pack(c, c);
    const float* row_buf = reinterpret_cast<const float*>(smem + kOffRow);
    const uint32_t t_s = tmem_addr(tmem_base, lane_base, kColBuf + 128 * grp), t_dp = t_s + 64;
    bool ok = true;
    int g = 0;  // steps of all items so far

    for (int w = 0;; ++w) {
        const int item = bars->ring.take(w, lane, abort_flag, kWaitLimitCycles);
        if (item < 0) {
            ok = (item == -1);
            break;
        }
        int kt, bh, s0, n;
        wk.get(item, &kt, &bh, &s0, &n);
        const int key = kt * kBlockK + r;
        for (int s = (g ^ grp) & 1; s < n; s += 2) {
            const int gs = g + s;
            const int rb = gs % kRowStages;
            ok = mbar_wait(&bars->row_full[rb], (gs / kRowStages) & 1, abort_flag);
            if (ok) ok = mbar_wait(&bars->sp_full[grp], (gs >> 1) & 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            const float4* l4 = reinterpret_cast<const float4*>(row_buf + rb * 2 * kStep);
            const float4* d4 = l4 + kStep / 4;
            // Keep key <= query.  Keys past the end of the sequence need no mask: their rows are not stored.
            const bool masked = kCausal && s < kBlockK / kStep;
            const int first = key - (s0 + s) * kStep;  // first kept query of the step
            // Half a step at a time, rolled: the two groups are at different places of this loop.
#pragma unroll 1
            for (int q = 0; q < kStep; q += 32) {
                uint32_t sv[32], dv[32], pk[16];
                tmem_ld_x32(t_s + q, sv);
                tmem_ld_x32(t_dp + q, dv);
                tmem_wait_ld();
                if (masked) {
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        if (q + i < first) sv[i] = 0xff800000u;  // -inf: P = 0
                }
#pragma unroll
                for (int i = 0; i < 32; i += 4) {
                    const float4 l = l4[(q + i) / 4];
                    float x0, x1, x2, x3;
                    f32x2_unpack(f32x2_fma(f32x2_pack(__uint_as_float(sv[i + 0]), __uint_as_float(sv[i + 1])), c2,
                                           f32x2_pack(l.x, l.y)), x0, x1);
                    f32x2_unpack(f32x2_fma(f32x2_pack(__uint_as_float(sv[i + 2]), __uint_as_float(sv[i + 3])), c2,
                                           f32x2_pack(l.z, l.w)), x2, x3);
                    x0 = ex2_approx(x0);
                    x1 = ex2_approx(x1);
                    x2 = ex2_approx(x2);
                    x3 = ex2_approx(x3);
                    pk[i / 2] = pack_bf16x2(x0, x1);
                    pk[i / 2 + 1] = pack_bf16x2(x2, x3);
                    // dS^T from the unrounded P^T: only what feeds a contraction is rounded (paper Section 4.3)
                    const float4 d = d4[(q + i) / 4];
                    f32x2_unpack(f32x2_mul(f32x2_pack(x0, x1), f32x2_add(f32x2_pack(__uint_as_float(dv[i + 0]),
                                                                                    __uint_as_float(dv[i + 1])),
                                                                         f32x2_pack(d.x, d.y))), x0, x1);
                    f32x2_unpack(f32x2_mul(f32x2_pack(x2, x3), f32x2_add(f32x2_pack(__uint_as_float(dv[i + 2]),
                                                                                    __uint_as_float(dv[i + 3])),
                                                                         f32x2_pack(d.z, d.w))), x2, x3);
                    dv[i / 2] = pack_bf16x2(x0, x1);
                    dv[i / 2 + 1] = pack_bf16x2(x2, x3);
                }
                tmem_st_x16(t_s + q / 2, pk);
                tmem_st_x16(t_dp + q / 2, dv);
            }
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&bars->ready[grp]);
                mbar_arrive(&bars->row_empty[rb]);
            }
        }
        if (!ok) break;
        g += n;
    }
}

// 128 bf16 numbers of key row r into a tile's two boxes, 128-byte swizzle.
__device__ __forceinline__ void kv_stage_row(uint8_t* stage, int r, const uint32_t (&pk)[D / 2]) {
#pragma unroll
    for (int x = 0; x < D / 8; ++x)
        *reinterpret_cast<uint4*>(stage + (x / 8) * kHalfTileBytes + r * 128 + (((x % 8) ^ (r & 7)) << 4)) =
            make_uint4(pk[4 * x], pk[4 * x + 1], pk[4 * x + 2], pk[4 * x + 3]);
}

// Write-out warps (warp `owarp` of four, thread = key row): dV, then dK * scale, of a finished item as bf16 into the item's K
// buffer and out with TMA stores, while the compute warps are in the next item.
template <bool kStrided>
__device__ __forceinline__ void kv_write_out(uint8_t* smem, KvBars* bars, uint32_t tmem_base, const CUtensorMap* tmdK,
                                             const CUtensorMap* tmdV, float scale, const KvWork& wk, int owarp, int lane) {
    volatile int* abort_flag = &bars->abort_flag;
    const uint32_t lane_base = 32u * owarp;
    const int r = lane_base + lane;
    const bool leader = (owarp == 0 && lane == 0);
    bool ok = true;
    for (int w = 0;; ++w) {
        const int item = bars->ring.take(w, lane, abort_flag, kWaitLimitCycles);
        if (item < 0) break;
        int kt, bh, s0, n;
        wk.get(item, &kt, &bh, &s0, &n);
        const int ks = w & 1;
        ok = mbar_wait(&bars->dkv_full, w & 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
        // Both go through the item's K buffer, dV first; dK waits in registers (64 of packed bf16) meanwhile, so that the
        // accumulators are free for the next item at once.
        const int hh = kStrided ? bh % wk.H : 0, bb = kStrided ? bh / wk.H : 0;
        uint8_t* stage = smem + kOffK + ks * kTileBytes;
        uint32_t pk[2][D / 2];
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
            if (which == 0) kv_stage_row(stage, r, pk[0]);
        }
        tc_fence_before();
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
            mbar_arrive(&bars->dkv_free);
            mbar_arrive(&bars->staged);
        }
        bool leader_ok = true;
        if (leader) {
            leader_ok = mbar_wait(&bars->staged, 0, abort_flag);
            if (leader_ok) {
#pragma unroll
                for (int h = 0; h < kHalves; ++h)
                    tma_store_tile<kStrided>(tmdV, stage + h * kHalfTileBytes, (wk.orders >> 20) & 15, h * kBoxCols,
                                             kt * kBlockK, hh, bb, bh);
                bulk_commit_group();
                bulk_wait_group_read<0>();
                mbar_arrive(&bars->stage_free);
            }
        }
        ok = __all_sync(0xffffffffu, leader_ok);
        if (ok) ok = mbar_wait(&bars->stage_free, w & 1, abort_flag);
        if (!ok) break;
        kv_stage_row(stage, r, pk[1]);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->staged);
        if (leader) {
            leader_ok = mbar_wait(&bars->staged, 1, abort_flag);
            if (leader_ok) {
#pragma unroll
                for (int h = 0; h < kHalves; ++h)
                    tma_store_tile<kStrided>(tmdK, stage + h * kHalfTileBytes, (wk.orders >> 16) & 15, h * kBoxCols,
                                             kt * kBlockK, hh, bb, bh);
                bulk_commit_group();
                bulk_wait_group_read<0>();
                mbar_arrive(&bars->k_empty[ks]);
            }
        }
        ok = __all_sync(0xffffffffu, leader_ok);
        if (!ok) break;
    }
    if (leader) bulk_wait_group<0>();  // dV and dK must be complete before the kernel ends
}

template <bool kCausal, bool kStrided>
__global__ void __launch_bounds__(kThreads, 1)
attn_dkdv_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                 const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmdO,
                 const __grid_constant__ CUtensorMap tmdK, const __grid_constant__ CUtensorMap tmdV,
                 const float* __restrict__ LSE, const float* __restrict__ Delta, int T, int BH, int H, uint32_t orders,
                 int n_tiles, int chunk, float scale, int* __restrict__ dev_status) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    if (smem != smem_raw) {
        // No room to realign: give up before anything is set up, but only once the predecessor in the stream
        // has completed (the status word is global memory, and this grid must not finish ahead of it).
        griddep_wait();
        if (threadIdx.x == 0) atomicExch(dev_status, kDevTimeout);
        return;
    }
    KvBars* bars = reinterpret_cast<KvBars*>(smem + kOffBar);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const KvWork wk{BH, n_tiles, chunk, T, H, orders, kCausal};

    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(&bars->k_full[s], 1);
            mbar_init(&bars->k_empty[s], 1);
            mbar_init(&bars->sp_full[s], 1);
            mbar_init(&bars->ready[s], 4);
        }
        for (int s = 0; s < kQStages; ++s) {
            mbar_init(&bars->q_full[s], 1);
            mbar_init(&bars->q_empty[s], 1);
        }
        for (int s = 0; s < kRowStages; ++s) {
            mbar_init(&bars->row_full[s], 1);
            mbar_init(&bars->row_empty[s], 4);
        }
        mbar_init(&bars->dkv_full, 1);
        mbar_init(&bars->dkv_free, 4);
        mbar_init(&bars->v_full, 1);
        mbar_init(&bars->v_empty, 1);
        mbar_init(&bars->staged, 4);
        mbar_init(&bars->stage_free, 1);
        mbar_init(&bars->drain, 1);
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
        if (lane == 0) kv_producer<kStrided>(&tmQ, &tmK, &tmV, &tmdO, smem, bars, wk);
    } else if (warp == 1) {
        kv_mma(smem, bars, tmem_base, wk);
    } else if (warp == 2) {
        kv_row_loader(bars, reinterpret_cast<float*>(smem + kOffRow), LSE, Delta, wk, lane);
    } else if (warp >= 12) {
        kv_write_out<kStrided>(smem, bars, tmem_base, &tmdK, &tmdV, scale, wk, warp & 3, lane);
    } else if (warp >= 4) {
        kv_compute<kCausal>(smem, bars, tmem_base, scale, wk, (warp - 4) >> 2, warp & 3, lane);
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, kTmemCols);
    if (threadIdx.x == 0 && bars->abort_flag != 0) atomicExch(dev_status, kDevTimeout);
}

}  // namespace

cudaError_t configure_attn_dkdv() {
    auto set = [](auto kernel) {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    };
    cudaError_t e = set(attn_dkdv_kernel<true, false>);
    if (e == cudaSuccess) e = set(attn_dkdv_kernel<true, true>);
    if (e == cudaSuccess) e = set(attn_dkdv_kernel<false, false>);
    if (e == cudaSuccess) e = set(attn_dkdv_kernel<false, true>);
    return e;
}

cudaError_t launch_attn_dkdv(const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV,
                             const CUtensorMap& tmdO, const CUtensorMap& tmdK, const CUtensorMap& tmdV, bool strided,
                             uint32_t orders, const float* LSE, const float* Delta, const AttnShape& s, int num_sms,
                             int* dev_status, cudaStream_t stream) {
    const int n_tiles = (s.T + kBlockK - 1) / kBlockK, BH = s.B * s.H;
    const int chunk = heads_per_chunk(BH, n_tiles, s.T, D, num_sms);
    const dim3 grid(static_cast<unsigned>(n_tiles) * BH);  // one CTA per item; those that do not start are taken over
    auto go = [&](auto kernel) {
        return launch_overlapped(kernel, grid, dim3(kThreads), kSmemBytes, stream, tmQ, tmK, tmV, tmdO, tmdK, tmdV, LSE, Delta,
                                 s.T, BH, s.H, orders, n_tiles, chunk, s.scale, dev_status);
    };
    if (s.causal) return strided ? go(attn_dkdv_kernel<true, true>) : go(attn_dkdv_kernel<true, false>);
    return strided ? go(attn_dkdv_kernel<false, true>) : go(attn_dkdv_kernel<false, false>);
}

}  // namespace nova
