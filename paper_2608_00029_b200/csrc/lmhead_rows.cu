// Loss head for a few rows (M <= 64: the last position of each of some sequences, a short prompt): the same
// outputs as lmhead.cu, on a kernel that is nothing but a stream over W.
//
// What bounds it is reading W once (77 MB at N = 50304, K = 768: 11.6 us at 6.65 TB/s); with so few rows the
// product itself is small.  The roles of the operands are therefore swapped: W supplies the 128 rows of an
// instruction and X its 16..64 columns, so no padding to 128 rows of X is loaded, multiplied or exponentiated,
// and a CTA's share of W is cut in tiles of equal height h (a multiple of 8, at most 128) such that every CTA gets
// the same number of tiles: 128-entry tiles on 148 CTAs would leave a third of them idle in the last round at
// N = 50304.  The ring holds eight tiles of W per SM (128 KB), enough to cover the latency of DRAM.
//
// Statistics: a thread of the epilogue holds one vocabulary entry of every row.  The maximum and the sum of a row
// are taken across the 32 lanes with the halving exchange (31 shuffles for 32 rows, and lane r ends up with
// the result of row r), carried from tile to tile by that lane, and merged over the four warps at the end: one
// (max, sum) pair per row and CTA instead of one per 128 entries, which the merge kernel below, a warp per row,
// reads in one go.
//
// 192 threads: warp 0 TMA producer, warp 1 UMMA issuer, warps 2-5 epilogue.
// N = 50304, K = 768, M = 24, logits stored, back to back from a graph, merge included: 18.7 us, against 45.7 us for
// lmhead_kernel (X padded to 128 rows, 256-entry tiles of W in two uneven rounds, 393 pairs per row merged by one
// block); lmhead_rows_plan says where that one is kept.
#include "../../include/nova_lmhead.h"
#include "kernels.h"
#include "ptx.cuh"

namespace nova {
namespace {

constexpr int kThreads = 192;
constexpr int kEpiWarps = 4;
constexpr int kTileV = 128;  // vocabulary entries of a tile, at most
constexpr int kBK = 64;      // k elements per stage
constexpr int kStages = 8;
constexpr int kWBytes = kTileV * kBK * 2;
constexpr int kXBytes = kLmHeadFewRows * kBK * 2;
constexpr int kStageBytes = kWBytes + kXBytes;
constexpr int kOffStat = kStages * kStageBytes;                              // float2 [kEpiWarps][kLmHeadFewRows]
constexpr int kOffTgt = kOffStat + kEpiWarps * kLmHeadFewRows * 8;           // int [kLmHeadFewRows]
constexpr int kOffBar = kOffTgt + kLmHeadFewRows * 4;
constexpr int kSmemBytes = kOffBar + 256 + 1024;
static_assert(kSmemBytes <= 232448, "exceeds the shared memory of one CTA");
constexpr int kTmemCols = 2 * kLmHeadFewRows;

struct Bars {
    uint64_t full[kStages], empty[kStages];
    uint64_t acc_full[2], acc_empty[2];
    uint64_t drain;
    uint32_t tmem_base;
    int abort_flag;
};
static_assert(sizeof(Bars) <= 256, "barrier block");

// Reduces v[0..31] over the 32 lanes by repeated halving: lane r returns op over all lanes of v[r].
template <typename Op>
__device__ __forceinline__ float reduce_columns(float (&v)[32], int lane, Op op) {
#pragma unroll
    for (int w = 16; w >= 1; w >>= 1) {
        const bool upper = (lane & w) != 0;
#pragma unroll
        for (int i = 0; i < w; ++i) {
            const float keep = upper ? v[i + w] : v[i];
            const float send = upper ? v[i] : v[i + w];
            v[i] = op(keep, __shfl_xor_sync(0xffffffffu, send, w));
        }
    }
    return v[0];
}

// kGroups: groups of 32 rows of X (1 or 2).
template <int kGroups>
__global__ void __launch_bounds__(kThreads, 1)
lmhead_rows_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW,
                   const int* __restrict__ targets, __nv_bfloat16* __restrict__ logits, float2* __restrict__ partials,
                   float* __restrict__ tgt_logit, int M, int N, int K, int m_pad, int tile_h,
                   int* __restrict__ dev_status) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    Bars* bars = reinterpret_cast<Bars*>(smem + kOffBar);
    float2* stat = reinterpret_cast<float2*>(smem + kOffStat);
    int* tgt_s = reinterpret_cast<int*>(smem + kOffTgt);
    volatile int* abort_flag = &bars->abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_tiles = (N + tile_h - 1) / tile_h;
    const int k_blocks = (K + kBK - 1) / kBK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&bars->full[s], 1);
            mbar_init(&bars->empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&bars->acc_full[b], 1);
            mbar_init(&bars->acc_empty[b], kEpiWarps);
        }
        mbar_init(&bars->drain, 1);
        bars->abort_flag = 0;
        fence_mbar_init();
        tma_prefetch_desc(&tmX);
        tma_prefetch_desc(&tmW);
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
    if (warp == 0 && lane == 0) {  // a ring's worth of this CTA's W on its way into L2 while the predecessor drains
        for (int s = 0; s < kStages; ++s)
            if (static_cast<int>(blockIdx.x) < n_tiles && s < k_blocks)
                tma_prefetch_2d(&tmW, s * kBK, static_cast<int>(blockIdx.x) * tile_h);
    }
    griddep_wait();

    if (warp == 0) {
        if (lane == 0) {
            int armed[kStages];
            for (int s = 0; s < kStages; ++s) armed[s] = -1;
            bool ok = true;
            int g = 0;  // k blocks loaded so far
            for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
                for (int kb = 0; kb < k_blocks; ++kb, ++g) {
                    const int s = g % kStages;
                    const uint32_t ph = (g / kStages) & 1;
                    ok = mbar_wait(&bars->empty[s], ph ^ 1, abort_flag);
                    if (!ok) break;
                    // tile_h rows of W and m_pad rows of X; what lies past N, M or K arrives as zeros.  Rows tile_h
                    // to 127 of the W tile keep what was there: they only reach accumulator lanes that nobody reads.
                    mbar_expect_tx(&bars->full[s], (tile_h + m_pad) * kBK * 2);
                    armed[s] = ph;
                    tma_load_2d(smem + s * kStageBytes, &tmW, &bars->full[s], kb * kBK, t * tile_h);
                    tma_load_2d(smem + s * kStageBytes + kWBytes, &tmX, &bars->full[s], kb * kBK, 0);
                }
            }
            if (!ok) {  // giving up: let the copies in flight land before the shared memory goes away
                int none = 0;
                for (int s = 0; s < kStages; ++s)
                    if (armed[s] >= 0) (void)mbar_wait(&bars->full[s], armed[s], &none);
            }
        }
    } else if (warp == 1) {
        // the whole warp in uniform control flow, one elected lane issues
        const uint32_t idesc = umma_idesc_bf16(kTileV, m_pad, 0, 0);
        const uint32_t hi = umma_desc_hi_sw128(1024);
        const bool el = elect_one();
        bool ok = true;
        int g = 0, it = 0;
        for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x, ++it) {
            const int ab = it & 1;
            ok = mbar_wait(&bars->acc_empty[ab], ((it >> 1) & 1) ^ 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            const uint32_t t_acc = tmem_base + ab * kLmHeadFewRows;
            for (int kb = 0; kb < k_blocks; ++kb, ++g) {
                const int s = g % kStages;
                ok = mbar_wait(&bars->full[s], (g / kStages) & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                if (el) {
                    const uint32_t a = umma_desc_lo(smem_u32(smem + s * kStageBytes), 16);
                    const uint32_t b = umma_desc_lo(smem_u32(smem + s * kStageBytes + kWBytes), 16);
#pragma unroll
                    for (int k = 0; k < kBK / 16; ++k)
                        umma_ss(t_acc, umma_desc_join(a + 2 * k, hi), umma_desc_join(b + 2 * k, hi), idesc,
                                (kb > 0 || k > 0) ? 1u : 0u);
                    tc_commit(&bars->empty[s]);
                    if (kb == k_blocks - 1) tc_commit(&bars->acc_full[ab]);
                }
                __syncwarp();
            }
        }
        if (!ok) {
            int none = 0;
            if (el) tc_commit(&bars->drain);
            __syncwarp();
            (void)mbar_wait(&bars->drain, 0, &none);
        }
    } else {
        const uint32_t lane_base = 32u * (warp & 3);
        const int ew = warp - 2, et = ew * 32 + lane;
        if (et < kLmHeadFewRows) tgt_s[et] = (et < M) ? targets[et] : -1;
        named_barrier_sync(1, kEpiWarps * 32);
        bool ok = true;
        int it = 0;
        // lane r: running maximum (base-2 units) and sum of rows r and 32 + r over this warp's entries
        float m2[kGroups], l[kGroups];
#pragma unroll
        for (int q = 0; q < kGroups; ++q) {
            m2[q] = -INFINITY;
            l[q] = 0.f;
        }
        for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x, ++it) {
            const int ab = it & 1;
            const int local = static_cast<int>(lane_base) + lane;
            const int v = t * tile_h + local;  // this thread's vocabulary entry
            const bool valid = local < tile_h && v < N;
            ok = mbar_wait(&bars->acc_full[ab], (it >> 1) & 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            const bool any = __any_sync(0xffffffffu, valid);
#pragma unroll
            for (int q = 0; q < kGroups; ++q) {
                if (32 * q >= M || !any) continue;
                uint32_t zr[32];
                __syncwarp();
                tmem_ld_x32(tmem_addr(tmem_base, lane_base, ab * kLmHeadFewRows + 32 * q), zr);
                tmem_wait_ld();
                if (q == kGroups - 1) {  // (columns past m_pad hold nothing that is used)
                    tc_fence_before();
                }
                if (valid) {
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        const int row = 32 * q + i;
                        if (tgt_s[row] == v) tgt_logit[row] = __uint_as_float(zr[i]);
                    }
                    if (logits != nullptr) {  // 32 consecutive entries of a row per warp and store
                        __nv_bfloat16* out = logits + static_cast<size_t>(32 * q) * N + v;
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            if (32 * q + i < M) out[static_cast<size_t>(i) * N] = __float2bfloat16_rn(__uint_as_float(zr[i]));
                    }
                }
                float z[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) z[i] = (valid && 32 * q + i < M) ? __uint_as_float(zr[i]) : -INFINITY;
                float tmp[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) tmp[i] = z[i];
                const float m_new = fmaxf(m2[q], reduce_columns(tmp, lane, [](float a, float b) { return fmaxf(a, b); }) * kLog2e);
                // rows past M stay at -inf: their reference is 0 and everything they add is 2^-inf = 0
                const float ref = (m_new == -INFINITY) ? 0.f : m_new;
#pragma unroll
                for (int i = 0; i < 32; ++i)
                    tmp[i] = ex2_approx(fmaf(z[i], kLog2e, -__shfl_sync(0xffffffffu, ref, i)));
                const float sum = reduce_columns(tmp, lane, [](float a, float b) { return a + b; });
                l[q] = l[q] * ex2_approx(m2[q] - ref) + sum;
                m2[q] = m_new;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->acc_empty[ab]);
        }
        // one pair per row for the whole CTA
#pragma unroll
        for (int q = 0; q < kGroups; ++q) stat[ew * kLmHeadFewRows + 32 * q + lane] = make_float2(m2[q], l[q]);
        named_barrier_sync(1, kEpiWarps * 32);
        if (et < M && ok) {
            float m = -INFINITY, s = 0.f;
            for (int w = 0; w < kEpiWarps; ++w) m = fmaxf(m, stat[w * kLmHeadFewRows + et].x);
            const float ref = (m == -INFINITY) ? 0.f : m;  // -inf: every logit of the CTA is (a masked stretch of the vocabulary)
            for (int w = 0; w < kEpiWarps; ++w) {
                const float2 p = stat[w * kLmHeadFewRows + et];
                s += p.y * ex2_approx(p.x - ref);
            }
            partials[static_cast<size_t>(et) * gridDim.x + blockIdx.x] = make_float2(m, s);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, kTmemCols);
    if (threadIdx.x == 0 && bars->abort_flag != 0) atomicExch(dev_status, kDevTimeout);
}

// Merge: a warp per row, the pairs of a row adjacent (at most kMergeSteps per lane, all loads in flight at once).
constexpr int kMergeWarps = 4, kMergeSteps = 8;

__global__ void __launch_bounds__(32 * kMergeWarps)
lmhead_rows_merge_kernel(const float2* __restrict__ partials, const float* __restrict__ tgt_logit,
                         const int* __restrict__ targets, float* __restrict__ lse, float* __restrict__ loss, int M, int N,
                         int n_part) {
    griddep_launch_dependents();
    griddep_wait();
    const int lane = threadIdx.x & 31;
    const int row = blockIdx.x * kMergeWarps + (threadIdx.x >> 5);
    if (row >= M) return;
    float2 p[kMergeSteps];
    float m = -INFINITY;
#pragma unroll
    for (int k = 0; k < kMergeSteps; ++k) {
        const int i = lane + 32 * k;
        p[k] = (i < n_part) ? partials[static_cast<size_t>(row) * n_part + i] : make_float2(-INFINITY, 0.f);
        m = fmaxf(m, p[k].x);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    const float ref = (m == -INFINITY) ? 0.f : m;
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < kMergeSteps; ++k) s += p[k].y * ex2_approx(p[k].x - ref);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) {
        const float v = m * kLn2 + logf(s);
        const int t = targets[row];
        lse[row] = v;
        loss[row] = (t >= 0 && t < N) ? v - tgt_logit[row] : 0.f;
    }
}

}  // namespace

cudaError_t configure_lmhead_rows() {
    cudaError_t e = cudaFuncSetAttribute(lmhead_rows_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(lmhead_rows_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
}

// When it pays.  This kernel against lmhead_kernel in us at N = 50304, K = 768, logits stored (part of W in L2): M = 24 15.0, 34.8;
// 48 22.9, 34.7; 64 23.3, 34.2, where the accumulator and the shuffles end.  Up to 32 rows it is the faster one at every N
// (1000 to 64000) and K (64 to 1600).  From 33 on a tile's epilogue has two groups of rows, which reading W has to pay for: not
// below some 5000 entries (N = 4096 0.92 to 1.10 of the other kernel's time, N = 8000 0.85 to 0.96), nor where a second
// round of tiles has only just begun and its tiles are low (N = 19000, tiles of 72: 0.74 to 1.14; N = 24000, tiles of 88:
// 0.64 to 0.97).
bool lmhead_rows_plan(int M, int N, int num_sms, int* ctas, int* tile_h, int* m_pad) {
    if (M > kLmHeadFewRows) return false;
    const int limit = num_sms < 32 * kMergeSteps ? num_sms : 32 * kMergeSteps;
    const int full = (N + kTileV - 1) / kTileV;  // also what the workspace has room for: one pair per row and 128 entries
    *ctas = full < limit ? full : limit;
    const int rounds = (full + *ctas - 1) / *ctas;
    const long long share = static_cast<long long>(*ctas) * rounds;
    *tile_h = static_cast<int>(((N + share - 1) / share + 7) / 8 * 8);
    const int n_tiles = (N + *tile_h - 1) / *tile_h;
    if (n_tiles < *ctas) *ctas = n_tiles;
    *m_pad = (M + 15) / 16 * 16;
    return M <= 32 || (N > 40 * kTileV && (rounds == 1 || *tile_h >= 88));
}

cudaError_t launch_lmhead_rows(const CUtensorMap& tmX, const CUtensorMap& tmW, const int* targets, void* logits,
                               float* lse, float* loss, int M, int N, int K, int ctas, int tile_h, int m_pad,
                               void* workspace, float* tgt_logit, int* dev_status, cudaStream_t stream) {
    float2* partials = static_cast<float2*>(workspace);
    auto go = [&](auto kernel) {
        return launch_overlapped(kernel, dim3(static_cast<unsigned>(ctas)), dim3(kThreads), kSmemBytes, stream, tmX, tmW,
                                 targets, static_cast<__nv_bfloat16*>(logits), partials, tgt_logit, M, N, K, m_pad,
                                 tile_h, dev_status);
    };
    const cudaError_t e = M <= 32 ? go(lmhead_rows_kernel<1>) : go(lmhead_rows_kernel<2>);
    if (e != cudaSuccess) return e;
    return launch_overlapped(lmhead_rows_merge_kernel, dim3((M + kMergeWarps - 1) / kMergeWarps), dim3(32 * kMergeWarps), 0,
                             stream, static_cast<const float2*>(partials), static_cast<const float*>(tgt_logit), targets,
                             lse, loss, M, N, ctas);
}

}  // namespace nova
