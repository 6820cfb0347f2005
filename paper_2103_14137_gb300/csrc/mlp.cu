// Candidate scorer of the learned proposal: a 3-layer perceptron
//   x (in) -> relu(x W1 + b1) (H) -> relu(. W2 + b2) (H) -> . w3 + b3 (logit)
// with BF16 weights and activations and FP32 accumulation, trained with
// binary cross-entropy on LP dwell-time labels (candidate kept by the relaxed
// LP (9) or not) and Adam.  The dense products run on the tensor cores
// (tcgen05.mma BF16 -> FP32, accumulator in tensor memory) through one GEMM
// tile that takes each operand along K or across it, so the forward pass, the
// weight gradients (X^T dZ) and the input gradients (dZ W^T) all use it.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <random>
#include <vector>

#include "tcgen05.cuh"
#include "uvc_internal.cuh"

struct uvc_mlp {
    int in_dim = 0, in_pad = 0, hidden = 0, max_batch = 0;
    int64_t step = 0;
    void* block = nullptr;
    // fp32 master parameters, gradients, Adam moments: one flat array each
    float *param = nullptr, *grad = nullptr, *m1 = nullptr, *m2 = nullptr;
    int64_t nparam = 0;
    float *W1, *b1, *W2, *b2, *w3, *b3;         // views into param
    __nv_bfloat16 *W1h, *W2h;                    // bf16 copies used by the GEMMs
    __nv_bfloat16 *Xh, *H1, *H2, *dZ1, *dZ2;     // activations, max_batch rows
    float *dS, *loss;                            // per row; loss[0] = the batch loss, the terms after it
    float *part, *cols;                          // partial sums of the gradients (GradArgs)
};

namespace uvc {
namespace {

// The GEMM on the fifth-generation tensor cores: one block per 128 x 64 tile of
// C, accumulated in tensor memory by tcgen05.mma .kind::f16 (BF16 operands,
// FP32 accumulator, M = 128, N = 64, K = 16 per instruction, K ascending).
// Every operand of the network is contiguous along one of its dimensions: along
// K (activations times weights) it is read in the tensor core's K-major layout,
// along M or N (weights forward; both operands of the weight gradients, whose K
// is the batch) in its MN-major layout, so either way 16 bytes of memory are
// 16 bytes of a core matrix and the tiles arrive by cp.async, zero-filled past
// the matrices' edges, two slices of 128 along K in flight (96 KB).  The first
// form gathered the operands element by element with a barrier and an MMA wait
// every 32 along K: 49-86 us for a forward product of a 4,096-row batch
// and 2,190-2,330 us for a weight gradient, one of 4 or 8 blocks walking 4,096
// rows each; the gradients are now split along the batch too.  Now 9 and
// 11 us forward, 16 us for all weight gradients and column sums; four training
// steps and their gradients read back 14.2 -> 0.29 ms (B = 4,096, 114-256-256-1).
// The epilogue reads the accumulator back with tcgen05.ld (warp w: rows
// 32w..32w+31).  A wait that runs out (bounded: about a second) makes the
// block write NaN.
constexpr int BM = 128, BN = 64, BK = 128, kGemmThreads = 128;
constexpr uint32_t kAStep = BM * 32, kBStep = BN * 32;              // bytes of one K-step (16 values)
constexpr uint32_t kAStage = (BK / 16) * kAStep, kBStage = (BK / 16) * kBStep;
constexpr uint32_t kGemmSmem = 2 * (kAStage + kBStage);
constexpr uint32_t kGemmTmemCols = BN;                              // FP32 accumulator columns

// Operand views: K-major A(m, k) = A[m lda + k], else A(m, k) = A[k lda + m];
// B likewise with n.  All extents along the contiguous dimension are multiples
// of 8 (hidden widths and padded inputs), and every row starts on 16 bytes.
struct GemmArgs {
    const __nv_bfloat16 *A, *B;
    int64_t lda, ldb;
    int M, N;
    int k0, k1;      // the slice of K to sum over
};

// One 16-byte chunk of an operand: `r8` along the 8 rows of a core matrix,
// (c, g) the chunk's place.  ROWS = M or N extent of the tile.
template <bool MN, int ROWS>
__device__ __forceinline__ void load_operand(const __nv_bfloat16* __restrict__ P, int64_t ld, int row0, int nrow, int k0,
                                             int k1, uint32_t smem) {
#pragma unroll
    for (int e = threadIdx.x; e < ROWS * (BK / 8); e += kGemmThreads) {
        const int r8 = e & 7;
        int64_t src;
        uint32_t off;
        bool in;
        if (MN) {   // chunk c of 8 rows (m or n), K group g of 8
            const int c = (e >> 3) % (ROWS / 8), g = (e >> 3) / (ROWS / 8);
            const int k = k0 + g * 8 + r8, r = row0 + c * 8;
            in = k < k1 && r < nrow;
            src = (int64_t)k * ld + r;
            off = (uint32_t)(g * (ROWS / 8) + c) * 128u + (uint32_t)r8 * 16u;
        } else {    // chunk c of 8 along K, row group g of 8
            const int c = (e >> 3) % (BK / 8), g = (e >> 3) / (BK / 8);
            const int k = k0 + c * 8, r = row0 + g * 8 + r8;
            in = k < k1 && r < nrow;
            src = (int64_t)r * ld + k;
            off = (uint32_t)(c >> 1) * (ROWS * 32) + (uint32_t)g * 256u + (uint32_t)(c & 1) * 128u + (uint32_t)r8 * 16u;
        }
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem + off), "l"(in ? P + src : P),
                     "r"(in ? 16 : 0)
                     : "memory");
    }
}

// The tile (m0, n0) of A B over [k0, k1): accumulated in tensor memory, handed
// to `out(m, n, v)` as 16 consecutive columns n..n + 15 of row m.
template <bool A_MN, bool B_MN, class Out>
__device__ __forceinline__ void gemm_tile(const GemmArgs& G, int m0, int n0, Out out) {
    extern __shared__ __align__(1024) unsigned char gemm_smem[];
    __shared__ uint64_t done[2];   // MMAs of the slices in buffer 0, 1
    __shared__ uint32_t tmem_slot;
    __shared__ int fail;
    constexpr uint32_t idesc = tc::idesc_f32acc(tc::kFmtBF16, BM, BN, A_MN, B_MN);
    constexpr uint32_t a_lbo = A_MN ? BM * 16 : 128, a_sbo = A_MN ? 128 : 256;
    constexpr uint32_t b_lbo = B_MN ? BN * 16 : 128, b_sbo = B_MN ? 128 : 256;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t base = tc::smem_u32(gemm_smem);
    const int nslice = (G.k1 - G.k0 + BK - 1) / BK;
    auto load = [&](int c) {
        const uint32_t buf = base + (uint32_t)(c & 1) * (kAStage + kBStage);
        load_operand<A_MN, BM>(G.A, G.lda, m0, G.M, G.k0 + c * BK, G.k1, buf);
        load_operand<B_MN, BN>(G.B, G.ldb, n0, G.N, G.k0 + c * BK, G.k1, buf + kAStage);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (nslice > 0) load(0);
    if (tid == 0) {
        fail = 0;
        tc::mbar_init(&done[0], 1);
        tc::mbar_init(&done[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tc::alloc(&tmem_slot, kGemmTmemCols);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = tmem_slot;
    for (int c = 0; c < nslice; ++c) {
        if (c + 1 < nslice) {   // the next slice's buffer is free once the MMAs of slice c - 1 are done
            if (c >= 1 && !fail && !tc::mbar_wait(&done[(c + 1) & 1], (uint32_t)((c - 1) >> 1) & 1u)) fail = 1;
            load(c + 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        tc::fence_proxy_async();
        __syncthreads();
        if (tid == 0) {
            tc::fence_after();
            const uint32_t a = base + (uint32_t)(c & 1) * (kAStage + kBStage), b = a + kAStage;
            const int steps = (min(BK, G.k1 - G.k0 - c * BK) + 15) / 16;
            for (int ks = 0; ks < steps; ++ks)
                tc::mma<false>(tmem, tc::smem_desc(a + ks * kAStep, a_lbo, a_sbo),
                               tc::smem_desc(b + ks * kBStep, b_lbo, b_sbo), idesc, (c > 0 || ks > 0) ? 1u : 0u);
            tc::commit(&done[c & 1]);
        }
    }
    // the last slice's commit covers every MMA before it
    if (nslice > 0 && !tc::mbar_wait(&done[(nslice - 1) & 1], (uint32_t)((nslice - 1) >> 1) & 1u)) fail = 1;
    __syncthreads();
    tc::fence_after();
    const bool bad = fail != 0;
    const int m = m0 + 32 * warp + lane;
#pragma unroll
    for (int c0 = 0; c0 < BN; c0 += 16) {
        float v[16];
        tc::load16(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)c0, v);
#pragma unroll
        for (int c = 0; c < 16; ++c) v[c] = bad ? __int_as_float(0x7fc00000) : (nslice > 0 ? v[c] : 0.f);
        if (m < G.M) out(m, n0 + c0, v);
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) {
        tc::fence_after();
        tc::dealloc(tmem, kGemmTmemCols);
    }
}

// 8 values as BF16, 16 bytes at p.
__device__ __forceinline__ void store8(__nv_bfloat16* p, const float* v) {
    __align__(16) __nv_bfloat16 h[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) h[q] = __float2bfloat16(v[q]);
    *reinterpret_cast<uint4*>(p) = *reinterpret_cast<const uint4*>(h);
}

// Y = relu(X W + b) in BF16: X [B][K], W [K][H].
__global__ void __launch_bounds__(kGemmThreads) k_layer(const __nv_bfloat16* __restrict__ X, int B, int K,
                                                        const __nv_bfloat16* __restrict__ W, int H,
                                                        const float* __restrict__ bias, __nv_bfloat16* __restrict__ Y) {
    const GemmArgs G{X, W, K, H, B, H, 0, K};
    gemm_tile<false, true>(G, blockIdx.x * BM, blockIdx.y * BN, [&](int m, int n, float (&v)[16]) {
#pragma unroll
        for (int h = 0; h < 16; h += 8) {
            if (n + h >= H) break;
            float y[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) y[q] = fmaxf(v[h + q] + bias[n + h + q], 0.f);
            store8(Y + (int64_t)m * H + n + h, y);
        }
    });
}

// dZ1 = (dZ2 W2^T) [H1 > 0] in BF16: dZ2 [B][H], W2 [H][H].
__global__ void __launch_bounds__(kGemmThreads) k_layer_back(const __nv_bfloat16* __restrict__ dZ2, int B, int H,
                                                             const __nv_bfloat16* __restrict__ W2,
                                                             const __nv_bfloat16* __restrict__ H1,
                                                             __nv_bfloat16* __restrict__ dZ1) {
    const GemmArgs G{dZ2, W2, H, H, B, H, 0, H};
    gemm_tile<false, false>(G, blockIdx.x * BM, blockIdx.y * BN, [&](int m, int n, float (&v)[16]) {
#pragma unroll
        for (int h = 0; h < 16; h += 8) {
            if (n + h >= H) break;
            const uint4 a4 = *reinterpret_cast<const uint4*>(H1 + (int64_t)m * H + n + h);
            const __nv_bfloat16* act = reinterpret_cast<const __nv_bfloat16*>(&a4);
            float y[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) y[q] = __bfloat162float(act[q]) > 0.f ? v[h + q] : 0.f;
            store8(dZ1 + (int64_t)m * H + n + h, y);
        }
    });
}

// The gradients that sum over the batch, in one launch.  Blocks [0, ngemm):
// gW1 = X^T dZ1 and gW2 = H1^T dZ2, a 128 x 64 tile and one of `nsplit` slices
// of the batch each (4 + 8 tiles of a 114 -> 256 -> 256 network would leave most
// of the chip idle); the rest: the column sums of dZ1, dZ2 and dS H2 (gb1, gb2,
// gw3) over one of `nchunk` row chunks, two columns a thread.  k_adam adds
// the partial results in a fixed order.
struct GradArgs {
    const __nv_bfloat16 *Xh, *H1, *H2, *dZ1, *dZ2;
    const float* dS;
    int B, P, H;
    int nsplit, per_split;      // batch slices of the products
    int nchunk, per_chunk;      // row chunks of the column sums
    float* part;                // [nsplit][P H + H H]
    float* cols;                // [3][nchunk][H]
};

__global__ void __launch_bounds__(kGemmThreads) k_weight_grads(GradArgs a, int tiles1, int tiles2, int tn) {
    const int ngemm = (tiles1 + tiles2) * a.nsplit;
    const int blk = blockIdx.x;
    if (blk < ngemm) {
        const int s = blk % a.nsplit, t = blk / a.nsplit;
        const bool first = t < tiles1;
        const int q = first ? t : t - tiles1;
        const GemmArgs G{first ? a.Xh : a.H1, first ? a.dZ1 : a.dZ2, first ? a.P : a.H, a.H, first ? a.P : a.H, a.H,
                         min(a.B, s * a.per_split), min(a.B, (s + 1) * a.per_split)};
        float* C = a.part + (size_t)s * ((size_t)a.P * a.H + (size_t)a.H * a.H) + (first ? 0 : (size_t)a.P * a.H);
        gemm_tile<true, true>(G, q / tn * BM, q % tn * BN, [&](int m, int n, float (&v)[16]) {
#pragma unroll
            for (int h = 0; h < 16; h += 4)
                if (n + h < a.H)
                    *reinterpret_cast<float4*>(C + (size_t)m * a.H + n + h) = make_float4(v[h], v[h + 1], v[h + 2], v[h + 3]);
        });
        return;
    }
    const int b = blk - ngemm, what = b % 3, chunk = b / 3;
    const __nv_bfloat16* X = what == 0 ? a.dZ1 : (what == 1 ? a.dZ2 : a.H2);
    const int r0 = chunk * a.per_chunk, r1 = min(a.B, r0 + a.per_chunk);
    for (int n = 2 * threadIdx.x; n < a.H; n += 2 * kGemmThreads) {
        float2 s = make_float2(0.f, 0.f);
#pragma unroll 8
        for (int i = r0; i < r1; ++i) {
            const float2 x = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(X + (int64_t)i * a.H + n));
            const float w = what == 2 ? a.dS[i] : 1.f;
            s.x += x.x * w;
            s.y += x.y * w;
        }
        *reinterpret_cast<float2*>(a.cols + ((size_t)what * a.nchunk + chunk) * a.H + n) = s;
    }
}

__global__ void k_to_bf16_pad(const float* __restrict__ x, int B, int in, int pad, __nv_bfloat16* __restrict__ y) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)B * pad) return;
    const int r = (int)(e / pad), c = (int)(e % pad);
    y[e] = __float2bfloat16(c < in ? x[(int64_t)r * in + c] : 0.f);
}

__global__ void k_cast_bf16(const float* __restrict__ x, int64_t n, __nv_bfloat16* __restrict__ y) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) y[e] = __float2bfloat16(x[e]);
}

// logit[i] = H2[i] . w3 + b3 (one warp per row)
__global__ void k_head(const __nv_bfloat16* __restrict__ H2, int B, int H, const float* __restrict__ w3,
                       const float* __restrict__ b3, float* __restrict__ logit) {
    const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (row >= B) return;
    float s = 0.f;
    for (int n = lane; n < H; n += 32) s += __bfloat162float(H2[(int64_t)row * H + n]) * w3[n];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) logit[row] = s + *b3;
}

// Training head, one warp per row: the logit (as k_head), then BCE with logits:
// dS = w (sigmoid(s) - y), the row's loss term, dZ2 = dS w3 [H2 > 0].
__global__ void k_head_back(const __nv_bfloat16* __restrict__ H2, int B, int H, const float* __restrict__ w3,
                            const float* __restrict__ b3, const float* __restrict__ y, const float* __restrict__ w,
                            float* __restrict__ dS, __nv_bfloat16* __restrict__ dZ2, float* __restrict__ loss_terms) {
    const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (row >= B) return;
    float s = 0.f;
    for (int n = lane; n < H; n += 32) s += __bfloat162float(H2[(int64_t)row * H + n]) * w3[n];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    s = __shfl_sync(0xffffffffu, s, 0) + *b3;
    const float p = 1.f / (1.f + expf(-s));
    const float d = w[row] * (p - y[row]);
    if (lane == 0) {
        dS[row] = d;
        const float sp = s > 0.f ? s + log1pf(expf(-s)) : log1pf(expf(s));   // softplus
        loss_terms[row] = w[row] * (sp - y[row] * s);
    }
    for (int n = lane; n < H; n += 32) {
        const float h = __bfloat162float(H2[(int64_t)row * H + n]);
        dZ2[(int64_t)row * H + n] = __float2bfloat16(h > 0.f ? d * w3[n] : 0.f);
    }
}

// Sum of x[0..n) by one block of 256 threads, fixed order; in thread 0.
__device__ float block_sum256(const float* __restrict__ x, int n) {
    __shared__ float part[256];
    float s = 0.f;
    for (int i = threadIdx.x; i < n; i += 256) s += x[i];
    __syncthreads();
    part[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) part[threadIdx.x] += part[threadIdx.x + o];
        __syncthreads();
    }
    return part[0];
}

struct AdamArgs {
    float *p, *g, *m, *v;
    __nv_bfloat16 *W1h, *W2h;
    float* loss;          // [1] and, after it, the B loss terms
    float* loss_out;      // the caller's, or null
    float lr, b1, b2, eps, c1, c2;
};

__device__ __forceinline__ float adam_update(const AdamArgs& A, int64_t e, float gi) {
    A.g[e] = gi;
    const float mi = A.b1 * A.m[e] + (1.f - A.b1) * gi;
    const float vi = A.b2 * A.v[e] + (1.f - A.b2) * gi * gi;
    A.m[e] = mi;
    A.v[e] = vi;
    return A.p[e] -= A.lr * (mi / A.c1) / (sqrtf(vi / A.c2) + A.eps);
}

// One thread per parameter: its gradient from the partial sums (fixed order),
// the Adam step, and the BF16 copy of a weight; the last block adds up dS (the
// gradient of b3) and the loss.
__global__ void __launch_bounds__(256) k_adam(AdamArgs A, GradArgs a) {
    const int64_t PH = (int64_t)a.P * a.H, HH = (int64_t)a.H * a.H, nw = PH + HH;
    if (blockIdx.x == gridDim.x - 1) {
        const float gb3 = block_sum256(a.dS, a.B);
        if (threadIdx.x == 0) adam_update(A, nw + 3 * (int64_t)a.H, gb3);
        const float loss = block_sum256(A.loss + 1, a.B);
        if (threadIdx.x == 0) {
            *A.loss = loss;
            if (A.loss_out) *A.loss_out = loss;
        }
        return;
    }
    const int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (e >= nw + 3 * (int64_t)a.H) return;
    const bool w1 = e < PH, w2 = e >= PH + a.H && e < nw + a.H;
    float g = 0.f;
    if (w1 || w2) {
        const float* q = a.part + (w1 ? e : e - a.H);
        for (int s = 0; s < a.nsplit; ++s) g += q[(size_t)s * nw];
    } else {
        const int64_t r = e < PH + a.H ? e - PH : a.H + (e - nw - a.H);   // b1, then b2 and w3
        const float* q = a.cols + r / a.H * a.nchunk * a.H + r % a.H;
        for (int c = 0; c < a.nchunk; ++c) g += q[(size_t)c * a.H];
    }
    const float p = adam_update(A, e, g);
    if (w1) A.W1h[e] = __float2bfloat16(p);
    if (w2) A.W2h[e - PH - a.H] = __float2bfloat16(p);
}

int blocks(int64_t n, int t = 256) { return (int)((n + t - 1) / t); }

void refresh_bf16(uvc_mlp* M, cudaStream_t s) {
    k_cast_bf16<<<blocks((int64_t)M->in_pad * M->hidden), 256, 0, s>>>(M->W1, (int64_t)M->in_pad * M->hidden, M->W1h);
    k_cast_bf16<<<blocks((int64_t)M->hidden * M->hidden), 256, 0, s>>>(M->W2, (int64_t)M->hidden * M->hidden, M->W2h);
}

// Dynamic shared memory above 48 KiB is opted into once per process.
cudaError_t gemm_smem_ok() {
    static const cudaError_t e = [] {
        cudaError_t r = cudaFuncSetAttribute(k_layer, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGemmSmem);
        if (r == cudaSuccess)
            r = cudaFuncSetAttribute(k_layer_back, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGemmSmem);
        if (r == cudaSuccess)
            r = cudaFuncSetAttribute(k_weight_grads, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGemmSmem);
        return r;
    }();
    return e;
}

dim3 tiles(int n, int m) { return dim3((m + BM - 1) / BM, (n + BN - 1) / BN); }

// Batch slices of the weight gradients: enough blocks to fill the chip, at
// most kMaxSplits partial copies, none shorter than one slice of K.
constexpr int kFillBlocks = 148, kMaxSplits = 16;
int grad_tiles(int P, int H) { return ((H + BN - 1) / BN) * ((P + BM - 1) / BM + (H + BM - 1) / BM); }
int max_splits(int P, int H) { return std::max(1, std::min(kMaxSplits, kFillBlocks / grad_tiles(P, H))); }
constexpr int kMaxChunks = 48;   // row chunks of the column sums

void hidden_layers(uvc_mlp* M, const float* x, int B, cudaStream_t s) {
    const int H = M->hidden, P = M->in_pad;
    k_to_bf16_pad<<<blocks((int64_t)B * P), 256, 0, s>>>(x, B, M->in_dim, P, M->Xh);
    k_layer<<<tiles(H, B), kGemmThreads, kGemmSmem, s>>>(M->Xh, B, P, M->W1h, H, M->b1, M->H1);
    k_layer<<<tiles(H, B), kGemmThreads, kGemmSmem, s>>>(M->H1, B, H, M->W2h, H, M->b2, M->H2);
}

void forward(uvc_mlp* M, const float* x, int B, float* logit, cudaStream_t s) {
    hidden_layers(M, x, B, s);
    k_head<<<blocks((int64_t)B * 32), 256, 0, s>>>(M->H2, B, M->hidden, M->w3, M->b3, logit);
}

}  // namespace
}  // namespace uvc

extern "C" {

int uvc_mlp_create(int32_t in_dim, int32_t hidden, int32_t max_batch, uint64_t seed, uvc_mlp** out) {
    if (!out) return UVC_E_INVAL;
    *out = nullptr;
    if (in_dim < 1 || in_dim > 4096 || hidden < 8 || hidden > 4096 || (hidden % 8) || max_batch < 1 ||
        max_batch > (1 << 24))
        return UVC_E_INVAL;
    uvc_mlp* M = new (std::nothrow) uvc_mlp();
    if (!M) return UVC_E_NOMEM;
    M->in_dim = in_dim;
    M->in_pad = (in_dim + 15) / 16 * 16;
    M->hidden = hidden;
    M->max_batch = max_batch;
    const int64_t P = M->in_pad, H = hidden, Bm = max_batch;
    M->nparam = P * H + H + H * H + H + H + 1;
    const size_t f4 = sizeof(float), h2 = sizeof(__nv_bfloat16);
    const size_t npart = (size_t)uvc::max_splits((int)P, (int)H) * (P * H + H * H);
    const size_t ncols = 3 * (size_t)uvc::kMaxChunks * H;
    size_t bytes = 4 * f4 * M->nparam + h2 * (P * H + H * H) + h2 * (Bm * P + 4 * Bm * H) +
                   f4 * (npart + ncols + 2 * Bm + 64) + 16 * 256;
    if (cudaMalloc(&M->block, bytes) != cudaSuccess) {
        cudaGetLastError();
        delete M;
        return UVC_E_NOMEM;
    }
    char* p = static_cast<char*>(M->block);
    auto take = [&](size_t n) {
        char* q = p;
        p += (n + 255) & ~size_t(255);
        return q;
    };
    M->param = (float*)take(f4 * M->nparam);
    M->grad = (float*)take(f4 * M->nparam);
    M->m1 = (float*)take(f4 * M->nparam);
    M->m2 = (float*)take(f4 * M->nparam);
    M->W1h = (__nv_bfloat16*)take(h2 * P * H);
    M->W2h = (__nv_bfloat16*)take(h2 * H * H);
    M->Xh = (__nv_bfloat16*)take(h2 * Bm * P);
    M->H1 = (__nv_bfloat16*)take(h2 * Bm * H);
    M->H2 = (__nv_bfloat16*)take(h2 * Bm * H);
    M->dZ1 = (__nv_bfloat16*)take(h2 * Bm * H);
    M->dZ2 = (__nv_bfloat16*)take(h2 * Bm * H);
    M->part = (float*)take(f4 * npart);
    M->cols = (float*)take(f4 * ncols);
    M->dS = (float*)take(f4 * Bm);
    M->loss = (float*)take(f4 * (Bm + 1));
    float* q = M->param;
    M->W1 = q; q += P * H; M->b1 = q; q += H; M->W2 = q; q += H * H; M->b2 = q; q += H; M->w3 = q; q += H; M->b3 = q;
    // He initialisation (padded input rows stay zero), zero biases
    std::vector<float> h(M->nparam, 0.f);
    std::mt19937_64 rng(seed);
    std::normal_distribution<float> n1(0.f, std::sqrt(2.f / in_dim)), n2(0.f, std::sqrt(2.f / hidden));
    for (int r = 0; r < in_dim; ++r)
        for (int c = 0; c < H; ++c) h[r * H + c] = n1(rng);
    for (int64_t e = 0; e < H * H; ++e) h[P * H + H + e] = n2(rng);
    for (int64_t e = 0; e < H; ++e) h[P * H + H + H * H + H + e] = n2(rng) * 0.5f;
    cudaError_t e = cudaMemcpy(M->param, h.data(), f4 * M->nparam, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(M->m1, 0, f4 * M->nparam);
    if (e == cudaSuccess) e = cudaMemset(M->m2, 0, f4 * M->nparam);
    if (e != cudaSuccess) {
        cudaFree(M->block);
        delete M;
        return uvc::status_from_cuda(e);
    }
    uvc::refresh_bf16(M, nullptr);
    e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        cudaFree(M->block);
        delete M;
        return uvc::status_from_cuda(e);
    }
    *out = M;
    return UVC_OK;
}

int uvc_mlp_free(uvc_mlp* M) {
    if (!M) return UVC_OK;
    cudaDeviceSynchronize();
    cudaFree(M->block);
    delete M;
    return UVC_OK;
}

int64_t uvc_mlp_param_count(const uvc_mlp* M) { return M ? M->nparam : -1; }

int uvc_mlp_params(uvc_mlp* M, float* host, int64_t n, int32_t set) {
    if (!M || !host || n != M->nparam) return UVC_E_INVAL;
    cudaError_t e = set ? cudaMemcpy(M->param, host, sizeof(float) * n, cudaMemcpyHostToDevice)
                        : cudaMemcpy(host, M->param, sizeof(float) * n, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && set) {
        uvc::refresh_bf16(M, nullptr);
        e = cudaDeviceSynchronize();
    }
    return uvc::status_from_cuda(e);
}

int uvc_mlp_forward(uvc_mlp* M, const float* x, int32_t B, float* logit, uvc_stream_t stream) {
    if (!M || B < 0 || B > M->max_batch || (B > 0 && (!x || !logit))) return UVC_E_INVAL;
    if (B == 0) return UVC_OK;
    const cudaError_t e = uvc::gemm_smem_ok();
    if (e != cudaSuccess) return uvc::status_from_cuda(e);
    uvc::forward(M, x, B, logit, (cudaStream_t)stream);
    return uvc::status_from_cuda(cudaGetLastError());
}

int uvc_mlp_train_step(uvc_mlp* M, const float* x, const float* y, const float* w, int32_t B, float lr,
                       float* loss, uvc_stream_t stream) {
    if (!M || B < 1 || B > M->max_batch || !x || !y || !w || !(lr > 0.f)) return UVC_E_INVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const int H = M->hidden, P = M->in_pad;
    cudaError_t e = uvc::gemm_smem_ok();
    if (e != cudaSuccess) return uvc::status_from_cuda(e);
    uvc::hidden_layers(M, x, B, s);
    uvc::k_head_back<<<uvc::blocks((int64_t)B * 32), 256, 0, s>>>(M->H2, B, H, M->w3, M->b3, y, w, M->dS, M->dZ2,
                                                                  M->loss + 1);
    uvc::k_layer_back<<<uvc::tiles(H, B), uvc::kGemmThreads, uvc::kGemmSmem, s>>>(M->dZ2, B, H, M->W2h, M->H1, M->dZ1);
    uvc::GradArgs a;
    a.Xh = M->Xh; a.H1 = M->H1; a.H2 = M->H2; a.dZ1 = M->dZ1; a.dZ2 = M->dZ2;
    a.dS = M->dS;
    a.B = B; a.P = P; a.H = H;
    a.per_split = (B + uvc::max_splits(P, H) - 1) / uvc::max_splits(P, H);
    a.per_split = std::max(uvc::BK, (a.per_split + 15) / 16 * 16);
    a.nsplit = (B + a.per_split - 1) / a.per_split;
    a.per_chunk = std::max(32, (B + uvc::kMaxChunks - 1) / uvc::kMaxChunks);
    a.nchunk = (B + a.per_chunk - 1) / a.per_chunk;
    a.part = M->part;
    a.cols = M->cols;
    const int tn = (H + uvc::BN - 1) / uvc::BN, t1 = tn * ((P + uvc::BM - 1) / uvc::BM),
              t2 = tn * ((H + uvc::BM - 1) / uvc::BM);
    uvc::k_weight_grads<<<(t1 + t2) * a.nsplit + 3 * a.nchunk, uvc::kGemmThreads, uvc::kGemmSmem, s>>>(a, t1, t2, tn);
    M->step += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - std::pow(b1, (float)M->step), c2 = 1.f - std::pow(b2, (float)M->step);
    const uvc::AdamArgs A{M->param, M->grad, M->m1, M->m2, M->W1h, M->W2h, M->loss, loss, lr, b1, b2, 1e-8f, c1, c2};
    uvc::k_adam<<<uvc::blocks(M->nparam - 1) + 1, 256, 0, s>>>(A, a);
    return uvc::status_from_cuda(cudaGetLastError());
}

int uvc_mlp_grads(const uvc_mlp* M, float* host, int64_t n) {
    if (!M || !host || n != M->nparam) return UVC_E_INVAL;
    return uvc::status_from_cuda(cudaMemcpy(host, M->grad, sizeof(float) * n, cudaMemcpyDeviceToHost));
}

}  // extern "C"
