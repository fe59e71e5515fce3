// Internal launch interface between the C ABI (api.cu) and the kernels.  Not installed.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace nova {

constexpr int kBlockQ = 128;        // query rows per tile (UMMA M)
constexpr int kBlockK = 128;        // keys per tile
constexpr int kBoxCols = 64;        // bf16 elements per 128-byte swizzled row (TMA box inner extent)
constexpr int kHalfTileBytes = 128 * 128;  // one [128 rows x 64 bf16] box

struct AttnShape {
    int B, H, T, D;
    int causal;
    float scale;
};

// Strides, in elements, of a bf16 tensor indexed [b, h, t, d]; d is contiguous.  [B,H,T,D] storage has
// (H*T*D, T*D, D); the Q slice of a fused projection output [B, T, 3, H, D] has (T*3*H*D, D, 3*H*D).
struct TensorStrides {
    long long b, h, t;
};

// Records a CUDA error code for nova_attn_last_cuda_error() of the calling thread and returns
// NOVA_ATTN_ERR_CUDA; for the entry points that live outside api.cu.
int record_cuda_error(int code);

// The argument checks every backward entry point makes before anything else (NULL pointers, shape, 16-byte
// alignment of the tensors, scale); returns NOVA_ATTN_OK or the error nova_attn_bwd would report.
int validate_bwd_args(const void* Q, const void* K, const void* V, const void* dO, const float* LSE,
                      const float* Delta, const void* dQ, const void* dK, const void* dV, int B, int H, int T, int D,
                      float scale);

// Launches `kernel` allowing it to overlap the tail of the previous kernel in `stream` (programmatic
// dependent launch); the kernel must call griddep_wait() before it touches global memory.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_overlapped(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem_bytes,
                                     cudaStream_t stream, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem_bytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Forward.  Two builds of every kernel.  Plain (`strided` false): all bf16 tensors have batch stride =
// H * head stride, so their maps are 3-D [D, T, B*H]; box of 64 x 128 tokens, 128-byte swizzle.  Strided:
// the maps are 4-D [D, x, y, z] with token / head / batch in order of increasing stride, and `orders`
// holds, four bits per tensor in the order Q, K, V, O, which of the three sits where (see
// tma_load_tile).  `tmO` describes the output and is used for TMA stores.  Persistent: launches at most
// `num_sms` CTAs.  `wait_limit`: cycle limit of every device-side wait; `inject`: test aid, 1 makes the
// loader leave out its first K-tile request so that a wait runs out (0 in normal use).
cudaError_t launch_attn_fwd(const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV,
                            const CUtensorMap& tmO, bool strided, uint32_t orders, float* LSE, const AttnShape& s,
                            int num_sms, long long wait_limit, int inject, int* dev_status, cudaStream_t stream);
cudaError_t configure_attn_fwd();

cudaError_t launch_attn_bwd_preprocess(const __nv_bfloat16* O, const __nv_bfloat16* dO, float* Delta,
                                       const AttnShape& s, const TensorStrides& so, const TensorStrides& sdo,
                                       int num_sms, cudaStream_t stream);

// The query-major passes of the backward (attn_dq.cu; dQ at D = 128 only): K and V maps with boxes of kKeyStep rows.
constexpr int kKeyStep = 64;
// Exact Delta_i = sum_j P_ij (dO_i . V_j) with P rebuilt from LSE (two contractions + exp2 per tile).
cudaError_t launch_attn_delta(const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV,
                              const CUtensorMap& tmdO, const float* LSE, float* Delta, const AttnShape& s,
                              int num_sms, int* dev_status, cudaStream_t stream);
// Deterministic dQ (the dQ half of the paper's two-kernel backward): one CTA per pair of 128-row query tiles walks
// the keys in order and writes dQ = bf16(scale * sum_j dS_j K_j) through `tmdQ`.  `strided`, `orders`: as in the
// forward, for Q, K, V, dO, dQ.
cudaError_t launch_attn_dq(const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV,
                           const CUtensorMap& tmdO, const CUtensorMap& tmdQ, bool strided, uint32_t orders,
                           const float* LSE, const float* Delta, const AttnShape& s, int num_sms, int* dev_status,
                           cudaStream_t stream);
cudaError_t configure_attn_dq();
// The same two at D = 64, with their operands in tensor memory (attn_dq64.cu).  The same bits of Delta.
cudaError_t launch_attn_delta64(const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV,
                                const CUtensorMap& tmdO, const float* LSE, float* Delta, const AttnShape& s, int* dev_status,
                                cudaStream_t stream);
cudaError_t launch_attn_dq64(const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV,
                             const CUtensorMap& tmdO, const CUtensorMap& tmdQ, bool strided, uint32_t orders,
                             const float* LSE, const float* Delta, const AttnShape& s, int* dev_status, cudaStream_t stream);
cudaError_t configure_attn_dq64();

// The dK/dV half of the two-kernel backward at D = 128 (attn_dkdv.cu): Q and dO maps with boxes of kKeyStep rows, the
// others of 128.  `orders` for Q, K, V, dO, dK, dV.
cudaError_t launch_attn_dkdv(const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV,
                             const CUtensorMap& tmdO, const CUtensorMap& tmdK, const CUtensorMap& tmdV, bool strided,
                             uint32_t orders, const float* LSE, const float* Delta, const AttnShape& s, int num_sms,
                             int* dev_status, cudaStream_t stream);
cudaError_t configure_attn_dkdv();
// The same at D = 64 (attn_dkdv64.cu).  `terms`: the row terms of every query as launch_row_terms64 leaves them (32 bytes for
// each of B * H * ceil(T / 64) * 64 rows, 16-byte aligned), or null: the kernel makes them itself (plain layout only).  Goes out
// right after the dQ kernel, whose end it does not wait for (ptx.cuh).
cudaError_t launch_row_terms64(const float* LSE, const float* Delta, void* terms, const AttnShape& s, cudaStream_t stream);
cudaError_t launch_attn_dkdv64(const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV,
                               const CUtensorMap& tmdO, const CUtensorMap& tmdK, const CUtensorMap& tmdV, bool strided,
                               uint32_t orders, const float* LSE, const float* Delta, const void* terms, const AttnShape& s,
                               int* dev_status, cudaStream_t stream);
cudaError_t configure_attn_dkdv64();

// Heads that the items of the kernels at D=128 are taken in together: enough items for two rounds of the SMs, and no more
// than about 48 MB of Q, K, V and dO, so that what the tiles of a head share stays in L2 (the forward re-reads K and V only,
// half of that).  All heads in one list, chunks, in us, forward / exact Delta / deterministic backward: B=16, H=32, T=1024
// 200, 174 / 173, 157 / 604, 547; B=4, H=32, T=2048 without the mask 280, 241 / 264, 240 / 908, 814.  Budgets of 24 and 96 MB
// are within 3 % of it, most within 1 %, in either direction (the forward at the first shape 184 and 176).  All heads where
// everything fits anyway (96 of the 126 MB): at 83 MB (B=16, H=16, T=333) 89.7 in one list, 92.2 us in two chunks, lost to
// the uneven end of the first; at 100 to 128 MB the two differ by at most 3 %.
inline int heads_per_chunk(int BH, int items_per_head, long long T, int D, int num_sms) {
    const long long per_head = T * D * 8;
    long long c = (48ll << 20) / per_head;
    const long long c_min = (2ll * num_sms + items_per_head - 1) / items_per_head;
    if (c < c_min) c = c_min;
    if (per_head * BH <= (96ll << 20) || c * 3 / 2 >= BH) return BH;
    const long long n = (BH + c - 1) / c;
    return static_cast<int>((BH + n - 1) / n);
}

// Steps after which the last SM is done with `items` work items that go out heaviest first, about: the longest item, or one
// item after another, the smallest of the first round with the largest of each later one.  steps(i): those of item i, with
// what an item costs besides.  For a few rounds of items (it adds them up).
template <typename F>
long long steps_until_done(long long items, int num_sms, F&& steps) {
    if (items <= num_sms) return steps(0);
    long long sum = steps(num_sms - 1);
    for (long long k = num_sms; k < items; k += num_sms) sum += steps(k);
    return steps(0) > sum ? steps(0) : sum;
}

// What the backward main kernel does with its partial tiles of dQ.
enum class DqMode {
    kAccumulate,  // adds them, unscaled, into the fp32 accumulator
    kDirect,      // T <= kBlockK, a head has one key tile: its dQ tile is complete and is written scaled, as bf16
};

// Backward main kernel: adds unscaled dQ partial tiles into the fp32 accumulator [B,H,T,D] (zero on
// entry) described by `tmAcc` (fp32 [D, T, B*H], box [32, 128, 1], 128-byte swizzle) and writes dK and dV
// through TMA stores (`tmdK`, `tmdV`: the bf16 maps of the outputs).  `strided`, `orders`: as in the forward, for
// Q, K, V, dO, dK, dV (and dQ).  `dq`: see above; `tmAcc` is the bf16 map of dQ with kDirect.
// Persistent: launches at most `num_sms` CTAs.
cudaError_t launch_attn_bwd(const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV,
                            const CUtensorMap& tmdO, const CUtensorMap& tmAcc, const CUtensorMap& tmdK,
                            const CUtensorMap& tmdV, bool strided, uint32_t orders, DqMode dq, const float* LSE,
                            const float* Delta, const AttnShape& s, int num_sms, int* dev_status, cudaStream_t stream);
cudaError_t configure_attn_bwd();

// Loss head (lmhead.cu): `tmX` is the 2-D map of X [K, M] with box [64, 128], `tmW` that of W [K, N] with box
// [64, 256], `tmL` that of the logits [N, M] with box [64, 32] (any valid map if `store_logits` is false), all
// bf16 with 128-byte swizzle.  Enqueues the fused contraction + statistics kernel and the merge.
cudaError_t launch_lmhead(const CUtensorMap& tmX, const CUtensorMap& tmW, const CUtensorMap& tmWh, const CUtensorMap& tmL,
                          bool store_logits, const int* targets, float* lse, float* loss, int M, int N, int K,
                          void* workspace, int num_sms, int* dev_status, cudaStream_t stream);
cudaError_t configure_lmhead();
size_t lmhead_workspace_bytes(int M, int N);
float* lmhead_target_logits(void* workspace, int M, int N);  // the part of the workspace behind the partial pairs
// Rows of the X and W boxes; returns the box width in k elements.
int lmhead_boxes(int* box_rows_x, int* box_rows_w);

// The same for at most kLmHeadFewRows rows (lmhead_rows.cu).  lmhead_rows_plan says whether this kernel is the faster one and
// chooses the number of CTAs, the height of a W tile (rows of the box of `tmW`) and the rows of the box of `tmX`; both boxes
// are 64 k elements wide.
constexpr int kLmHeadFewRows = 64;
cudaError_t configure_lmhead_rows();
bool lmhead_rows_plan(int M, int N, int num_sms, int* ctas, int* tile_h, int* m_pad);
cudaError_t launch_lmhead_rows(const CUtensorMap& tmX, const CUtensorMap& tmW, const int* targets, void* logits,
                               float* lse, float* loss, int M, int N, int K, int ctas, int tile_h, int m_pad,
                               void* workspace, float* tgt_logit, int* dev_status, cudaStream_t stream);

// Clears `bytes` (a multiple of 16) at the 16-byte aligned `ptr`.
cudaError_t launch_zero(void* ptr, size_t bytes, int num_sms, cudaStream_t stream);

// dQ = bf16(scale * dq_acc); the accumulator is contiguous [B,H,T,D], dQ has strides `sdq`.
cudaError_t launch_dq_convert(const float* dq_acc, __nv_bfloat16* dQ, const AttnShape& s, const TensorStrides& sdq,
                              float scale, int num_sms, cudaStream_t stream);

}  // namespace nova
