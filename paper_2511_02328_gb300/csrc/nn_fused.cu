// nn_fused.cu -- the classifier's inference in one kernel: one cluster of two,
// four or eight blocks per image, every activation in shared memory (the
// layered path of model.cu, which keeps the activations for the backward pass,
// serves training).
//
// Same network and precision policy: input bf16 [64][64][2]; three blocks
// conv3x3 (pad 1) + bias -> ReLU -> 2x2 max pool, 2 -> 16 -> 32 -> 64
// channels, the pooled activations rounded to bf16; global average pool,
// FC 64 -> 2, softmax.  Weights are rounded from the fp32 master parameters to
// bf16 (nearest even) in shared memory.
//
// Each convolution is an implicit GEMM on mma.sync.m16n8k16 (bf16 -> fp32):
// an M tile is a 2 x 8 pixel patch (rows g and g + 8 of the fragment are the
// vertically adjacent pixels (y, x) and (y + 1, x), x = 8 tx + g), so a 2x2
// pool window sits in one thread (vertical pair) and its neighbour lane
// g ^ 1 (horizontal pair, one shuffle); A fragments are read straight from
// the NHWC activations (a 32-bit word = two consecutive input channels of one
// tap, k = (dy * 3 + dx) * cin + i), B fragments from the packed weights
// [cout][K].  Bias, ReLU, pooling and the bf16 rounding happen in the
// accumulator registers.
//
// Block r of a cluster of CL owns image rows 64 / CL r .. and the rows they pool to
// in every layer, and keeps only those and a halo row on either side; a layer's
// first and last row are also written into the neighbours' halos through
// distributed shared memory.  Each block rounds its share of the weights of
// layers 2 and 3 and writes it into all of the cluster's.  Pixels and rows of
// weights are padded so that a warp's fragment loads fall in distinct banks.
// Every pixel's sums are the same whatever CL is.
// Bound by latency (a chain of loads, three layers and four cluster barriers).
// A call on 1 / 16 / 36 / 76 / 152 / 255 images took 42 / 42 / 41 / 41 / 44 / 77 us
// with one block per image (which rounded all 23,000 weights and ran every tile
// alone), and takes 10 / 14 / 14 / 19 / 25 / 45 us.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "internal.h"
#include "nn.h"

namespace cg = cooperative_groups;

namespace {

constexpr int FT = 256;          // threads (8 warps)
constexpr int S1 = 24, S2 = 40;                 // elements per pixel of the block 1 and 2 outputs (16 and 32 used)
constexpr int K1 = 32, K2 = 144, K3 = 288;      // padded K of each conv (9 cin rounded up to 16)
constexpr int P1 = K1 + 8, P2 = K2 + 8, P3 = K3 + 8;  // elements per row of packed weights
constexpr int W1_E = 16 * P1, W2_E = 32 * P2, W3_E = 64 * P3;
constexpr int NF = 16 + 32 + 64 + 128 + 2 + 64 + 2;   // biases, fw, fb, gap, logits (floats)

// Shared-memory layout (bf16 elements) of a block of a cluster of CL: its rows
// of each activation with halo rows and columns, then the weights.
template <int CL>
struct Lay {
    static constexpr int R0 = 64 / CL, R1 = 32 / CL, R2 = 16 / CL, R3 = 8 / CL;  // own rows of the input and the outputs
    static constexpr int IN_E = (R0 + 2) * 66 * 2;      // input rows R0 r - 1 .. R0 r + R0
    static constexpr int A1_E = (R1 + 2) * 34 * S1;     // block 1 output
    static constexpr int A2_E = (R2 + 2) * 18 * S2;     // block 2 output
    static constexpr int A3_E = 8 * 8 * 64;             // block 3 output, whole, gathered in block 0 (over its block 1
                                                        // output, which no block reads any more)
    static constexpr int IN = 0, A1 = (IN + IN_E + 7) / 8 * 8, A2 = A1 + A1_E, A3 = A1;
    static constexpr int W1 = A2 + A2_E, W2 = W1 + W1_E, W3 = W2 + W2_E, END = W3 + W3_E;
    static_assert(A1_E % 8 == 0 && A2_E % 8 == 0 && W1_E % 8 == 0 && W2_E % 8 == 0 && W3_E % 8 == 0, "16-byte parts");
    static_assert(A3_E <= A1_E, "the block 3 output fits over the block 1 output");
    static constexpr size_t BYTES = (size_t)END * 2 + (size_t)NF * 4;
};

__device__ __forceinline__ uint32_t ld32(const __nv_bfloat16* p) { return *reinterpret_cast<const uint32_t*>(p); }

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// conv3x3 + bias + ReLU + 2x2 max pool of a block's PR pooled rows.  in: local
// rows with halo, (W + 2) pixels of CS elements; w: [COUT][KP].  A work unit is
// one 2 x 8 pixel tile and UN of its COUT / 8 column groups.  Pooled values go
// to put(local pooled row, pooled column, channel, two channels).
template <int CIN, int CS, int COUT, int W, int KS, int KP, int PR, int UN, typename Put>
__device__ __forceinline__ void conv_band(const __nv_bfloat16* in, const __nv_bfloat16* w, const float* bias, Put&& put)
{
    constexpr int TX = W / 8, NG = COUT / 8 / UN, UNITS = PR * TX * NG;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
    for (int t = warp; t < UNITS; t += FT / 32) {
        const int n0 = t % NG * UN, tx = t / NG % TX, ty = t / NG / TX;
        const int y0 = 2 * ty, x = 8 * tx + g;
        float acc[UN][4];
#pragma unroll
        for (int nt = 0; nt < UN; nt++)
#pragma unroll
            for (int e = 0; e < 4; e++) acc[nt][e] = 0.f;
#pragma unroll
        for (int ks = 0; ks < KS; ks++) {
            uint32_t a[4];
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int kk = ks * 16 + 2 * q + 8 * h;
                const int pos = kk / CIN, i = kk % CIN;
                if (pos < 9) {
                    const int dy = pos / 3, dx = pos % 3;
                    a[2 * h] = ld32(in + ((y0 + dy) * (W + 2) + x + dx) * CS + i);
                    a[2 * h + 1] = ld32(in + ((y0 + 1 + dy) * (W + 2) + x + dx) * CS + i);
                } else {
                    a[2 * h] = a[2 * h + 1] = 0u;
                }
            }
#pragma unroll
            for (int nt = 0; nt < UN; nt++) {
                const __nv_bfloat16* wr = w + ((n0 + nt) * 8 + g) * KP + ks * 16 + 2 * q;
                mma_bf16(acc[nt], a, ld32(wr), ld32(wr + 8));
            }
        }
#pragma unroll
        for (int nt = 0; nt < UN; nt++) {
            const int col = (n0 + nt) * 8 + 2 * q;
            float v0 = fmaxf(fmaxf(acc[nt][0] + bias[col], 0.f), fmaxf(acc[nt][2] + bias[col], 0.f));
            float v1 = fmaxf(fmaxf(acc[nt][1] + bias[col + 1], 0.f), fmaxf(acc[nt][3] + bias[col + 1], 0.f));
            v0 = fmaxf(v0, __shfl_xor_sync(0xffffffffu, v0, 4));
            v1 = fmaxf(v1, __shfl_xor_sync(0xffffffffu, v1, 4));
            if ((g & 1) == 0) put(ty, x >> 1, col, __floats2bfloat162_rn(v0, v1));
        }
    }
}

__device__ __forceinline__ void st2(__nv_bfloat16* p, __nv_bfloat162 v) { *reinterpret_cast<__nv_bfloat162*>(p) = v; }

template <int CL>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(FT)
k_forward_fused(const __nv_bfloat16* __restrict__ x, const float* __restrict__ w0, const float* __restrict__ b0,
                const float* __restrict__ w1, const float* __restrict__ b1, const float* __restrict__ w2,
                const float* __restrict__ b2, const float* __restrict__ fw, const float* __restrict__ fb,
                float* __restrict__ logits, float* __restrict__ prob)
{
    using L = Lay<CL>;
    extern __shared__ __align__(16) uint8_t smem[];
    __nv_bfloat16* S = reinterpret_cast<__nv_bfloat16*>(smem);
    float* F = reinterpret_cast<float*>(smem + (size_t)L::END * 2);
    float *sb0 = F, *sb1 = F + 16, *sb2 = F + 48, *sfw = F + 112, *sfb = F + 240, *gap = F + 242, *lg = F + 306;
    cg::cluster_group cluster = cg::this_cluster();
    const int tid = threadIdx.x, r = (int)cluster.block_rank();
    const int img = blockIdx.x / CL;

    // this block's share of the layer 2 and 3 weights, 8 at a time: 18 and 36 groups per row of K2 and K3
    constexpr int G2 = 32 * (K2 / 8), GALL = G2 + 64 * (K3 / 8), GB = GALL / CL;
    static_assert(GALL % CL == 0, "whole shares");
    constexpr int GT = (GB + FT - 1) / FT;
    float4 wv[GT][2];
    int wo[GT];
#pragma unroll
    for (int k = 0; k < GT; k++) {
        const int e = tid + k * FT, gi = r * GB + e;
        wo[k] = -1;
        if (e < GB) {
            const bool two = gi < G2;
            const int o = two ? gi / (K2 / 8) : (gi - G2) / (K3 / 8), c = two ? gi % (K2 / 8) : (gi - G2) % (K3 / 8);
            const float4* src = reinterpret_cast<const float4*>(two ? w1 + o * K2 + 8 * c : w2 + o * K3 + 8 * c);
            wv[k][0] = __ldg(src);
            wv[k][1] = __ldg(src + 1);
            wo[k] = two ? L::W2 + o * P2 + 8 * c : L::W3 + o * P3 + 8 * c;
        }
    }
    // the block's input rows and one on either side (zero outside the image and in the halo columns)
    const uint32_t* xi = reinterpret_cast<const uint32_t*>(x + (int64_t)img * 64 * 64 * 2);
    uint32_t* in = reinterpret_cast<uint32_t*>(S + L::IN);
    for (int p = tid; p < (L::R0 + 2) * 66; p += FT) {
        const int y = L::R0 * r - 1 + p / 66, c = p % 66 - 1;
        in[p] = y >= 0 && y < 64 && c >= 0 && c < 64 ? __ldg(xi + y * 64 + c) : 0u;
    }
    // zero halos (and padding) of the layer outputs
    uint4* Z = reinterpret_cast<uint4*>(S + L::A1);
    for (int i = tid; i < (L::A1_E + L::A2_E) / 8; i += FT) Z[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int e = tid; e < 16 * K1; e += FT) {
        const int o = e / K1, k = e % K1;
        S[L::W1 + o * P1 + k] = __float2bfloat16_rn(k < 18 ? __ldg(w0 + o * 18 + k) : 0.f);
    }
    if (tid < 16) sb0[tid] = __ldg(b0 + tid);
    if (tid < 32) sb1[tid] = __ldg(b1 + tid);
    if (tid < 64) sb2[tid] = __ldg(b2 + tid);
    if (tid < 128) sfw[tid] = __ldg(fw + tid);
    if (tid < 2) sfb[tid] = __ldg(fb + tid);
    cluster.sync();  // every block runs and has zeroed its buffers

#pragma unroll
    for (int k = 0; k < GT; k++)
        if (wo[k] >= 0) {
            uint4 v;
            const __nv_bfloat162 h[4] = {
                __floats2bfloat162_rn(wv[k][0].x, wv[k][0].y), __floats2bfloat162_rn(wv[k][0].z, wv[k][0].w),
                __floats2bfloat162_rn(wv[k][1].x, wv[k][1].y), __floats2bfloat162_rn(wv[k][1].z, wv[k][1].w)};
            v.x = reinterpret_cast<const uint32_t&>(h[0]);
            v.y = reinterpret_cast<const uint32_t&>(h[1]);
            v.z = reinterpret_cast<const uint32_t&>(h[2]);
            v.w = reinterpret_cast<const uint32_t&>(h[3]);
#pragma unroll
            for (int q = 0; q < CL; q++) *reinterpret_cast<uint4*>(cluster.map_shared_rank(S + wo[k], q)) = v;
        }

    // a layer's pooled row p goes to local row p + 1 here; the first also to the
    // previous block's last halo row, the last also to the next block's first
    __nv_bfloat16* up = r > 0 ? cluster.map_shared_rank(S, r - 1) : nullptr;
    __nv_bfloat16* down = r < CL - 1 ? cluster.map_shared_rank(S, r + 1) : nullptr;
    conv_band<2, 2, 16, 64, K1 / 16, P1, L::R1, 2>(
        S + L::IN, S + L::W1, sb0, [&](int p, int c, int ch, __nv_bfloat162 v) {
            const int o = (c + 1) * S1 + ch;
            st2(S + L::A1 + (p + 1) * 34 * S1 + o, v);
            if (p == 0 && up) st2(up + L::A1 + (L::R1 + 1) * 34 * S1 + o, v);
            if (p == L::R1 - 1 && down) st2(down + L::A1 + o, v);
        });
    cluster.sync();
    conv_band<16, S1, 32, 32, K2 / 16, P2, L::R2, 4>(
        S + L::A1, S + L::W2, sb1, [&](int p, int c, int ch, __nv_bfloat162 v) {
            const int o = (c + 1) * S2 + ch;
            st2(S + L::A2 + (p + 1) * 18 * S2 + o, v);
            if (p == 0 && up) st2(up + L::A2 + (L::R2 + 1) * 18 * S2 + o, v);
            if (p == L::R2 - 1 && down) st2(down + L::A2 + o, v);
        });
    cluster.sync();
    __nv_bfloat16* A3 = cluster.map_shared_rank(S, 0) + L::A3 + r * L::R3 * 8 * 64;
    conv_band<32, S2, 64, 16, K3 / 16, P3, L::R3, 2 * L::R3 >= 8 ? 8 : 2 * L::R3>(
        S + L::A2, S + L::W3, sb2, [&](int p, int c, int ch, __nv_bfloat162 v) { st2(A3 + (p * 8 + c) * 64 + ch, v); });
    cluster.sync();
    if (r != 0) return;

    // global average pool (fixed order), FC, softmax
    if (tid < 64) {
        float acc = 0.f;
#pragma unroll 16
        for (int p = 0; p < 64; p++) acc += __bfloat162float(S[L::A3 + p * 64 + tid]);
        gap[tid] = acc / 64.f;
    }
    __syncthreads();
    if (tid < 2) {
        float v = sfb[tid];
#pragma unroll 16
        for (int i = 0; i < 64; i++) v += gap[i] * sfw[tid * 64 + i];
        lg[tid] = v;
    }
    __syncthreads();
    if (tid == 0) {
        const float mx = fmaxf(lg[0], lg[1]);
        const float e0 = expf(lg[0] - mx), e1 = expf(lg[1] - mx);
        logits[2 * img] = lg[0];
        logits[2 * img + 1] = lg[1];
        if (prob) prob[img] = e1 / (e0 + e1);
    }
}

}  // namespace

namespace {

template <int CL, typename... Args>
int launch_fused(int n, cudaStream_t s, Args... args)
{
    if (int rc = af_ensure_smem((const void*)k_forward_fused<CL>, Lay<CL>::BYTES)) return rc;
    k_forward_fused<CL><<<n * CL, FT, Lay<CL>::BYTES, s>>>(args...);
    return af_cuda_check(cudaGetLastError(), "fused forward launch");
}

}  // namespace

int nn_forward_fused(const __nv_bfloat16* x, int n, const float* w0, const float* b0, const float* w1,
                     const float* b1, const float* w2, const float* b2, const float* fw, const float* fb,
                     float* logits, float* prob, cudaStream_t s)
{
    if (n <= 0) return AF_OK;
    // As many blocks per image as the SMs hold one each: a call of 8 / 4 / 2 blocks per image took 10.6 / 14.1 / 18.5 us
    // on 6 images, 16.4 / 14.4 / 18.5 us on 36 and 30.8 / 26.6 / 18.5 us on 76 (GB300, 152 SMs).
    int dev = 0, nsm = 0;
    AF_CUDA(cudaGetDevice(&dev));
    AF_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    if (8 * n <= nsm) return launch_fused<8>(n, s, x, w0, b0, w1, b1, w2, b2, fw, fb, logits, prob);
    if (4 * n <= nsm) return launch_fused<4>(n, s, x, w0, b0, w1, b1, w2, b2, fw, fb, logits, prob);
    return launch_fused<2>(n, s, x, w0, b0, w1, b1, w2, b2, fw, fb, logits, prob);
}
