// Memory-bound helpers of the backward pass.
//   bwd_preprocess_kernel: Delta_i = sum_d dO[i,d] * O[i,d]   (row term of the softmax Jacobian)
//   dq_convert_kernel:     dQ = bf16(scale * fp32 accumulator)
//   zero_kernel:           clears the fp32 accumulator before the backward kernel adds into it
// Both stream their inputs once with 16-byte loads; rows are split over D/8 lanes and reduced with
// xor-shuffles.  Grids are sized in multiples of the SM count.  The bf16 tensors may be strided
// (batch, head and token strides in elements, multiples of 8): a row index r = (b*H + h)*T + t is
// then split again; the contiguous case skips that arithmetic.
#include "kernels.h"
#include "ptx.cuh"

namespace nova {
namespace {

__device__ __forceinline__ float dot8_bf16(const uint4& a, const uint4& b) {
    const __nv_bfloat162* pa = reinterpret_cast<const __nv_bfloat162*>(&a);
    const __nv_bfloat162* pb = reinterpret_cast<const __nv_bfloat162*>(&b);
    float acc = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 fa = __bfloat1622float2(pa[i]);
        const float2 fb = __bfloat1622float2(pb[i]);
        acc = fmaf(fa.x, fb.x, acc);
        acc = fmaf(fa.y, fb.y, acc);
    }
    return acc;
}

// n / d for 0 <= n < 2^31 without a division instruction (Granlund and Montgomery, "Division by Invariant Integers using
// Multiplication", 1994): with 2^(s-1) < d <= 2^s and m = floor(2^32 (2^s - d) / d) + 1 the quotient is
// (umulhi(n, m) + n) >> s, and the sum stays below 2^32.
struct FastDiv {
    uint32_t m, s, d;
    explicit FastDiv(int divisor) : m(0), s(0), d(static_cast<uint32_t>(divisor)) {
        while ((1ull << s) < d) ++s;
        m = static_cast<uint32_t>(((1ull << 32) * ((1ull << s) - d)) / d + 1);
    }
    __device__ __forceinline__ uint32_t div(uint32_t n) const { return (__umulhi(n, m) + n) >> s; }
};

// How a row index r = (b*H + h)*T + t is split again for strided tensors.
struct RowSplit {
    FastDiv T, H;
    int wide;  // 2^31 rows or more
};

// Offset, in 16-byte units, of row r of a tensor with strides `s`.
__device__ __forceinline__ long long row_offset16(long long r, const RowSplit& rs, const TensorStrides& s) {
    uint32_t t, b, h;
    if (rs.wide) {
        const long long bh = r / rs.T.d;
        t = static_cast<uint32_t>(r - bh * rs.T.d);
        b = static_cast<uint32_t>(bh / rs.H.d);
        h = static_cast<uint32_t>(bh - static_cast<long long>(b) * rs.H.d);
    } else {
        const uint32_t r32 = static_cast<uint32_t>(r), bh = rs.T.div(r32);
        t = r32 - bh * rs.T.d;
        b = rs.H.div(bh);
        h = bh - b * rs.H.d;
    }
    return (b * s.b + h * s.h + t * s.t) >> 3;
}

// LPR = lanes per row = D/8 (8 for D=64, 16 for D=128); each lane owns 8 consecutive bf16.
template <int LPR, int UNROLL, bool kContiguous>
__global__ void __launch_bounds__(256) bwd_preprocess_kernel(const uint4* __restrict__ O, const uint4* __restrict__ dO,
                                                             float* __restrict__ Delta, long long rows, const RowSplit rs,
                                                             const TensorStrides so, const TensorStrides sdo) {
    griddep_launch_dependents();
    griddep_wait();
    const long long tid = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    const long long nthreads = static_cast<long long>(gridDim.x) * blockDim.x;
    const long long rows_per_pass = nthreads / LPR;
    const int sub = static_cast<int>(tid % LPR);
    long long r = tid / LPR;
    for (; r < rows; r += rows_per_pass * UNROLL) {
        uint4 a[UNROLL], b[UNROLL];
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
            const long long ru = r + u * rows_per_pass;
            if (ru < rows) {
                a[u] = __ldg(O + (kContiguous ? ru * LPR : row_offset16(ru, rs, so)) + sub);
                b[u] = __ldg(dO + (kContiguous ? ru * LPR : row_offset16(ru, rs, sdo)) + sub);
            } else {
                a[u] = make_uint4(0, 0, 0, 0);
                b[u] = make_uint4(0, 0, 0, 0);
            }
        }
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
            float acc = dot8_bf16(a[u], b[u]);
#pragma unroll
            for (int off = LPR / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
            const long long ru = r + u * rows_per_pass;
            if (sub == 0 && ru < rows) Delta[ru] = acc;
        }
    }
}

// Heads inside tokens (O and dO as [B,T,H,D] views): a block takes a tile of tokens of kTokHeads heads, reads them in the order
// in which they lie in memory, kTokHeads * 2 * D bytes at a time, and turns the sums round in shared memory, so that
// Delta [B,H,T] is written in lines as well.  Of 8, 4 and 2 heads the number that pads H least (8 alone left most lanes
// of a model with two or three heads idle: H=2, B=32, T=2048, D=64 15.4 us against 5.5, 8.4 head by head).  A thread has
// kBatches * 4 rows, four in flight: one batch, so that small problems have more blocks (B=1, H=12, T=1024, D=128 3.9 us with
// two, 2.3 with one), but two at D=128 from six blocks per SM on (B=8, H=32, T=1024: 26.2 us with one, 25.1 with two).
// Head by head through such a layout (128 bytes every 2 KB) reading took 8.4 us at B=8, H=16, T=1024, D=64 and 15.8 us at
// B=4, H=32, T=1000, D=128, against 5.5 and 9.4 us here (inputs in L2); from DRAM 16.4 and 24.6 against 14.3 and 21.4.
__host__ __device__ constexpr int tok_tile(int D, int heads, int batches) { return batches * 4 * (2048 / D) / heads; }

template <int LPR, int kTokHeads, int kBatches>
__global__ void __launch_bounds__(256, 4) bwd_preprocess_tokens_kernel(const uint4* __restrict__ O, const uint4* __restrict__ dO,
                                                                    float* __restrict__ Delta, int H, int T, int t_tiles,
                                                                    int h_tiles, const TensorStrides so,
                                                                    const TensorStrides sdo) {
    constexpr int kRowsPerPass = 256 / LPR, kPasses = 4, kTokTile = tok_tile(8 * LPR, kTokHeads, kBatches);
    __shared__ float sums[kTokHeads][kTokTile + 1];
    griddep_launch_dependents();
    const int h0 = static_cast<int>(blockIdx.x) % h_tiles * kTokHeads;
    const int bt = static_cast<int>(blockIdx.x) / h_tiles, t0 = bt % t_tiles * kTokTile;
    const long long b = bt / t_tiles;
    const int sub = threadIdx.x % LPR, row0 = threadIdx.x / LPR;
    const uint4* po = O + ((b * so.b) >> 3) + sub;
    const uint4* pd = dO + ((b * sdo.b) >> 3) + sub;
    griddep_wait();
#pragma unroll
    for (int p = 0; p < kBatches * kPasses; p += kPasses) {
        uint4 x[kPasses], y[kPasses];
#pragma unroll
        for (int u = 0; u < kPasses; ++u) {
            const int r = row0 + (p + u) * kRowsPerPass, t = t0 + r / kTokHeads, h = h0 + r % kTokHeads;
            x[u] = y[u] = make_uint4(0, 0, 0, 0);
            if (t < T && h < H) {
                x[u] = __ldg(po + ((h * so.h + t * so.t) >> 3));
                y[u] = __ldg(pd + ((h * sdo.h + t * sdo.t) >> 3));
            }
        }
#pragma unroll
        for (int u = 0; u < kPasses; ++u) {
            float acc = dot8_bf16(x[u], y[u]);
#pragma unroll
            for (int off = LPR / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
            const int r = row0 + (p + u) * kRowsPerPass;
            if (sub == 0) sums[r % kTokHeads][r / kTokHeads] = acc;
        }
    }
    __syncthreads();
    if (threadIdx.x >= kTokTile * kTokHeads) return;
    const int h = h0 + threadIdx.x / kTokTile, t = t0 + threadIdx.x % kTokTile;
    if (h < H && t < T) Delta[(b * H + h) * T + t] = sums[threadIdx.x / kTokTile][threadIdx.x % kTokTile];
}

// Each thread takes kConvertItems groups of 8 elements per pass and issues all their loads before the
// first store.
constexpr int kConvertItems = 4;

template <bool kContiguous>
__global__ void __launch_bounds__(256) dq_convert_kernel(const float4* __restrict__ acc, uint4* __restrict__ dQ,
                                                         long long n8, float scale, int lpr_shift, const RowSplit rs,
                                                         const TensorStrides sdq) {
    griddep_launch_dependents();
    griddep_wait();
    const long long stride = static_cast<long long>(gridDim.x) * blockDim.x * kConvertItems;
    for (long long base = static_cast<long long>(blockIdx.x) * blockDim.x * kConvertItems + threadIdx.x; base < n8;
         base += stride) {
        float4 a[kConvertItems], b[kConvertItems];
#pragma unroll
        for (int k = 0; k < kConvertItems; ++k) {
            const long long i = base + static_cast<long long>(k) * blockDim.x;
            if (i < n8) {
                a[k] = __ldcs(acc + 2 * i);
                b[k] = __ldcs(acc + 2 * i + 1);
            }
        }
#pragma unroll
        for (int k = 0; k < kConvertItems; ++k) {
            const long long i = base + static_cast<long long>(k) * blockDim.x;
            if (i >= n8) continue;
            uint4 v;
            v.x = pack_bf16x2(a[k].x * scale, a[k].y * scale);
            v.y = pack_bf16x2(a[k].z * scale, a[k].w * scale);
            v.z = pack_bf16x2(b[k].x * scale, b[k].y * scale);
            v.w = pack_bf16x2(b[k].z * scale, b[k].w * scale);
            if (kContiguous) {
                dQ[i] = v;
            } else {
                const long long r = i >> lpr_shift;
                dQ[row_offset16(r, rs, sdq) + (i - (r << lpr_shift))] = v;
            }
        }
    }
}

__global__ void __launch_bounds__(256) zero_kernel(uint4* __restrict__ p, long long n16) {
    griddep_launch_dependents();
    griddep_wait();
    const long long stride = static_cast<long long>(gridDim.x) * blockDim.x;
    for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < n16; i += stride)
        p[i] = make_uint4(0, 0, 0, 0);
}

}  // namespace

cudaError_t launch_zero(void* ptr, size_t bytes, int num_sms, cudaStream_t stream) {
    constexpr int kThreads = 256;
    const long long n16 = static_cast<long long>(bytes / 16);
    long long blocks = (n16 + kThreads - 1) / kThreads;
    const long long cap = static_cast<long long>(num_sms) * 8;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    return launch_overlapped(zero_kernel, dim3(static_cast<unsigned>(blocks)), dim3(kThreads), 0, stream,
                             static_cast<uint4*>(ptr), n16);
}

namespace {
RowSplit split_of(const AttnShape& s) {
    return RowSplit{FastDiv(s.T), FastDiv(s.H), static_cast<long long>(s.B) * s.H * s.T >= (1ll << 31) ? 1 : 0};
}
bool is_contiguous(const AttnShape& s, const TensorStrides& st) {
    return st.t == s.D && st.h == static_cast<long long>(s.T) * s.D && st.b == static_cast<long long>(s.H) * s.T * s.D;
}
}  // namespace

cudaError_t launch_attn_bwd_preprocess(const __nv_bfloat16* O, const __nv_bfloat16* dO, float* Delta,
                                       const AttnShape& s, const TensorStrides& so, const TensorStrides& sdo,
                                       int num_sms, cudaStream_t stream) {
    constexpr int kThreads = 256, kUnroll = 4;
    const long long rows = static_cast<long long>(s.B) * s.H * s.T;
    const int lpr = s.D / 8;
    const long long rows_per_block = kThreads / lpr * kUnroll;
    long long blocks = (rows + rows_per_block - 1) / rows_per_block;
    const long long cap = static_cast<long long>(num_sms) * 8;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    const uint4* o4 = reinterpret_cast<const uint4*>(O);
    const uint4* d4 = reinterpret_cast<const uint4*>(dO);
    const dim3 grid(static_cast<unsigned>(blocks));
    const bool contiguous = is_contiguous(s, so) && is_contiguous(s, sdo);
    if (!contiguous && so.h < so.t && sdo.h < sdo.t) {
        int heads = 8;
        auto padded = [&](int n) { return (s.H + n - 1) / n * n; };
        for (int n : {4, 2})
            if (padded(n) < padded(heads)) heads = n;
        const long long rows_padded = static_cast<long long>(s.B) * padded(heads) * s.T;
        const int batches = (s.D == 128 && rows_padded / (128 * 6) >= num_sms) ? 2 : 1;
        const int tile = tok_tile(s.D, heads, batches), t_tiles = (s.T + tile - 1) / tile, h_tiles = (s.H + heads - 1) / heads;
        const long long blocks_tok = static_cast<long long>(s.B) * t_tiles * h_tiles;
        auto go = [&](auto kernel) {
            return launch_overlapped(kernel, dim3(static_cast<unsigned>(blocks_tok)), dim3(kThreads), 0, stream, o4, d4, Delta,
                                     s.H, s.T, t_tiles, h_tiles, so, sdo);
        };
        if (blocks_tok <= 0x7fffffff) {
            if (s.D == 64)
                return heads == 8   ? go(bwd_preprocess_tokens_kernel<8, 8, 1>)
                       : heads == 4 ? go(bwd_preprocess_tokens_kernel<8, 4, 1>)
                                    : go(bwd_preprocess_tokens_kernel<8, 2, 1>);
            if (batches == 1)
                return heads == 8   ? go(bwd_preprocess_tokens_kernel<16, 8, 1>)
                       : heads == 4 ? go(bwd_preprocess_tokens_kernel<16, 4, 1>)
                                    : go(bwd_preprocess_tokens_kernel<16, 2, 1>);
            return heads == 8   ? go(bwd_preprocess_tokens_kernel<16, 8, 2>)
                   : heads == 4 ? go(bwd_preprocess_tokens_kernel<16, 4, 2>)
                                : go(bwd_preprocess_tokens_kernel<16, 2, 2>);
        }
    }
    auto go = [&](auto kernel) {
        return launch_overlapped(kernel, grid, dim3(kThreads), 0, stream, o4, d4, Delta, rows, split_of(s), so, sdo);
    };
    if (s.D == 64) return contiguous ? go(bwd_preprocess_kernel<8, kUnroll, true>) : go(bwd_preprocess_kernel<8, kUnroll, false>);
    return contiguous ? go(bwd_preprocess_kernel<16, kUnroll, true>) : go(bwd_preprocess_kernel<16, kUnroll, false>);
}

cudaError_t launch_dq_convert(const float* dq_acc, __nv_bfloat16* dQ, const AttnShape& s, const TensorStrides& sdq,
                              float scale, int num_sms, cudaStream_t stream) {
    constexpr int kThreads = 256;
    const long long n8 = static_cast<long long>(s.B) * s.H * s.T * s.D / 8;  // D is a multiple of 8
    long long blocks = (n8 + kThreads * kConvertItems - 1) / (kThreads * kConvertItems);
    const long long cap = static_cast<long long>(num_sms) * 8;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    const int lpr_shift = (s.D == 64) ? 3 : 4;
    const dim3 grid(static_cast<unsigned>(blocks));
    auto go = [&](auto kernel) {
        return launch_overlapped(kernel, grid, dim3(kThreads), 0, stream, reinterpret_cast<const float4*>(dq_acc),
                                 reinterpret_cast<uint4*>(dQ), n8, scale, lpr_shift, split_of(s), sdq);
    };
    return is_contiguous(s, sdq) ? go(dq_convert_kernel<true>) : go(dq_convert_kernel<false>);
}

}  // namespace nova
