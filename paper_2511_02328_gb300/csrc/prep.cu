// prep.cu -- preprocessing of the filterbank before the search (Sec. 2.2):
// square-law time downsampling and the zero-DM filter.
//
//   out[c][k] = min( sqrt(V * S / N), V ),  S = sum of bin k (N samples), V = 255,
//   rounded half up, exactly: floor((isqrt(floor(4 V S / N)) + 1) / 2) (below).
//
// Downsampling by 4, 8, 16 or 32 of rows of whole 16-byte pieces takes its bins straight
// from 16-byte loads (k_downsample4); any other factor or alignment goes through
// shared memory, one block per (channel, run of bins).  HBM-bound: nchan * nsamp
// bytes read, nchan * nsamp / D written.  The zero-DM filter of up to 4096 channels
// holds a tile of every channel in the shared memory of a thread-block cluster and
// reads the input once; wider inputs are read twice.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "internal.h"

namespace cg = cooperative_groups;

namespace {

constexpr int kDsThreads = 256;
constexpr int kDsSpan = 32768;  // bytes of input per block (shared memory)

// The rounded square root floor((isqrt(floor(T / N)) + 1) / 2), T = 4 V S, without
// an integer division: isqrt(floor(T / N)) = max r with r^2 N <= T.  A float
// estimate (rcpN = 1/N) is within one of r; two exact integer tests settle it.
__device__ __forceinline__ uint32_t sqlaw_value(uint64_t T, uint32_t N, float rcpN)
{
    uint32_t r = (uint32_t)sqrtf((float)T * rcpN);
    if ((uint64_t)r * r * N > T) r--;
    if ((uint64_t)(r + 1) * (r + 1) * N <= T) r++;
    const uint32_t v = (r + 1) / 2;
    return v < 255u ? v : 255u;
}

// floor((isqrt(floor(T / N)) + 1) / 2) = the largest v with (2 v - 1)^2 N <= T
// (v >= 1; else 0), in 32 bits for D <= 16384 (T = 1020 S < 2^32, (2 v - 1)^2 N <=
// 511^2 * 16384 < 2^32): an approximate square root, rounded up by more than
// its error (510 * 2^-21), is that v or the next, and one integer test decides.
__device__ __forceinline__ uint32_t sqlaw_value32(uint32_t S, uint32_t N, float scale)  // scale = 1020 / N
{
    float y;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(y) : "f"((float)S * scale));
    uint32_t v = (uint32_t)fmaf(y, 0.5f, 0.501f);
    const uint32_t r = 2u * v - 1u;
    if (v > 0u && r * r * N > 1020u * S) v--;
    return v;
}

// Sum of the n bytes from byte p of the shared words (n >= 1).
__device__ __forceinline__ uint32_t byte_sum(const uint32_t* w32, int p, int n)
{
    int w = p >> 2;
    const int e = p + n, we = e >> 2;  // the last word may be partial
    uint32_t S = 0;
    if (p & 3) {
        uint32_t x = w32[w] & (0xFFFFFFFFu << (8 * (p & 3)));
        if (w == we) return __dp4a(x & ~(0xFFFFFFFFu << (8 * (e & 3))), 0x01010101u, 0u);
        S = __dp4a(x, 0x01010101u, S);
        w++;
    }
    for (; w < we; w++) S = __dp4a(w32[w], 0x01010101u, S);
    if (e & 3) S = __dp4a(w32[w] & ~(0xFFFFFFFFu << (8 * (e & 3))), 0x01010101u, S);
    return S;
}

// Any D and alignment.  Block = (channel, run of tb bins).  The run's input is
// read as the aligned 16-byte pieces that hold it, wherever the row starts (rows
// of a length that is no multiple of 16 start off a boundary), all of a thread's
// loads issued first; byte mis + i of the shared array is the run's byte i.
__global__ void __launch_bounds__(kDsThreads)
k_downsample(const uint8_t* __restrict__ X, int64_t nsamp, int64_t total, int D, int64_t nout, int tb, unsigned runs,
             uint8_t* __restrict__ out)
{
    __shared__ __align__(16) uint8_t sx[kDsSpan + 32];
    const int c = (int)(blockIdx.x / runs);
    const int64_t k0 = (int64_t)(blockIdx.x % runs) * tb;
    const int64_t t0 = k0 * D;
    const int span = (int)min((int64_t)tb * D, nsamp - t0);
    const uint8_t* x = X + (int64_t)c * nsamp + t0;
    const int mis = (int)(reinterpret_cast<uintptr_t>(x) & 15);
    const uint8_t* xa = x - mis;
    const int n16 = (mis + span + 15) >> 4;
    {
        constexpr int NB = kDsSpan / 16 / kDsThreads + 1;
        // pieces wholly inside the input (those at its two ends may not be)
        const int lo = xa < X ? 1 : 0;
        const int hi = (int)min((int64_t)n16, ((int64_t)(X + total - xa)) >> 4);
        uint4 v[NB];
#pragma unroll
        for (int u = 0; u < NB; u++) {
            const int i = (int)threadIdx.x + u * kDsThreads;
            if (i >= lo && i < hi) v[u] = __ldg(reinterpret_cast<const uint4*>(xa) + i);
        }
#pragma unroll
        for (int u = 0; u < NB; u++) {
            const int i = (int)threadIdx.x + u * kDsThreads;
            if (i >= lo && i < hi) reinterpret_cast<uint4*>(sx)[i] = v[u];
        }
        if (lo > 0)
            for (int i = mis + (int)threadIdx.x; i < 16 && i < mis + span; i += kDsThreads) sx[i] = __ldg(xa + i);
        if (hi < n16)
            for (int i = max(mis, 16 * max(hi, lo)) + (int)threadIdx.x; i < mis + span; i += kDsThreads)
                sx[i] = __ldg(xa + i);
    }
    __syncthreads();
    const uint32_t* w32 = reinterpret_cast<const uint32_t*>(sx);
    const float rD = 1020.0f / (float)D;
    const int nb = (int)min((int64_t)tb, nout - k0);
    uint8_t* o = out + (int64_t)c * nout + k0;
    for (int k = (int)threadIdx.x; k < nb; k += kDsThreads) {
        const int a = k * D, n = min(D, span - a);
        const uint32_t S = byte_sum(w32, mis + a, n);
        o[k] = (uint8_t)(D <= 16384 ? sqlaw_value32(S, (uint32_t)n, n == D ? rD : 1020.0f / (float)n)
                                    : sqlaw_value(4ull * 255ull * S, (uint32_t)n, 1.0f / (float)n));
    }
}

// D = 4 Q with Q = 1, 2, 4 or 8, rows of whole 16-byte pieces: four bins are Q
// pieces, which a thread reads straight into registers (kDsG groups of four
// bins, all loads first) and answers with one 4-byte store; no shared memory.
// Bound by HBM and issue.  4096 x 2^18, D = 8: 0.42 ms through shared memory, with an
// IEEE square root and two integer tests per bin; 0.17 ms so.
constexpr int kDsG = 4;
template <int Q>
__global__ void __launch_bounds__(kDsThreads)
k_downsample4(const uint8_t* __restrict__ X, int64_t nsamp, int64_t nout, unsigned runs, uint8_t* __restrict__ out)
{
    constexpr int D = 4 * Q;
    const int c = (int)(blockIdx.x / runs);
    const int64_t g0 = (int64_t)(blockIdx.x % runs) * (kDsThreads * kDsG) + threadIdx.x;  // groups of four bins
    const uint8_t* x = X + (int64_t)c * nsamp;
    uint8_t* o = out + (int64_t)c * nout;
    const int64_t full = nsamp / (4 * D);  // groups of four whole bins
    uint4 v[kDsG][Q];
#pragma unroll
    for (int u = 0; u < kDsG; u++) {
        const int64_t g = g0 + u * kDsThreads;
        if (g < full) {
#pragma unroll
            for (int i = 0; i < Q; i++) v[u][i] = __ldg(reinterpret_cast<const uint4*>(x) + g * Q + i);
        }
    }
    const bool words = (reinterpret_cast<uintptr_t>(o) & 3) == 0;
#pragma unroll
    for (int u = 0; u < kDsG; u++) {
        const int64_t g = g0 + u * kDsThreads;
        if (g < full) {
            uint32_t word = 0;
#pragma unroll
            for (int j = 0; j < 4; j++) {
                uint32_t S = 0;
#pragma unroll
                for (int i = 0; i < Q; i++) {
                    const int q = j * Q + i;  // word of the group
                    const uint4& p = v[u][q >> 2];
                    S = __dp4a((q & 3) == 0 ? p.x : (q & 3) == 1 ? p.y : (q & 3) == 2 ? p.z : p.w, 0x01010101u, S);
                }
                word |= sqlaw_value32(S, D, 1020.0f / (float)D) << (8 * j);
            }
            if (words) {
                *reinterpret_cast<uint32_t*>(o + 4 * g) = word;
            } else {
#pragma unroll
                for (int j = 0; j < 4; j++) o[4 * g + j] = (uint8_t)(word >> (8 * j));
            }
        } else {  // the row's last bins (at most four, the last may be short)
            for (int64_t k = 4 * g; k < min(nout, 4 * g + 4); k++) {
                const int n = (int)min((int64_t)D, nsamp - k * D);
                uint32_t S = 0;
                for (int i = 0; i < n; i++) S += __ldg(x + k * D + i);
                o[k] = (uint8_t)sqlaw_value32(S, (uint32_t)n, 1020.0f / (float)n);
            }
        }
    }
}

template <int Q>
int launch_downsample4(const uint8_t* d_in, int nchan, int64_t nsamp, int64_t nout, uint8_t* d_out, cudaStream_t s)
{
    const int64_t runs = (nout + 4 * kDsThreads * kDsG - 1) / (4 * kDsThreads * kDsG);
    if ((long double)runs * nchan > 0x7fffffff) return af_set_error(AF_EINVAL, "af_downsample: input too large");
    k_downsample4<Q><<<(unsigned)(runs * nchan), kDsThreads, 0, s>>>(d_in, nsamp, nout, (unsigned)runs, d_out);
    return af_cuda_check(cudaGetLastError(), "af_downsample launch");
}

}  // namespace

extern "C" int af_downsample(const uint8_t* d_in, int nchan, int64_t nsamp, int D, uint8_t* d_out, void* stream)
try {
    if (!d_in || !d_out) return af_set_error(AF_EINVAL, "af_downsample: NULL buffer");
    if (nchan < 1 || nsamp < 1) return af_set_error(AF_EINVAL, "af_downsample: empty input");
    if (D < 1 || D > kDsSpan) return af_set_error(AF_EINVAL, "af_downsample: D %d not in 1..%d", D, kDsSpan);
    const int64_t nout = (nsamp + D - 1) / D;
    const int tb = kDsSpan / D;
    const int64_t runs = (nout + tb - 1) / tb;
    if ((long double)runs * nchan > 0x7fffffff) return af_set_error(AF_EINVAL, "af_downsample: input too large");
    // four bins in whole 16-byte pieces of aligned rows: through registers
    if (nsamp % 16 == 0 && (uintptr_t)d_in % 16 == 0) {
        cudaStream_t st = (cudaStream_t)stream;
        if (D == 4) return launch_downsample4<1>(d_in, nchan, nsamp, nout, d_out, st);
        if (D == 8) return launch_downsample4<2>(d_in, nchan, nsamp, nout, d_out, st);
        if (D == 16) return launch_downsample4<4>(d_in, nchan, nsamp, nout, d_out, st);
        if (D == 32) return launch_downsample4<8>(d_in, nchan, nsamp, nout, d_out, st);
    }
    k_downsample<<<(unsigned)(runs * nchan), kDsThreads, 0, (cudaStream_t)stream>>>(d_in, nsamp, nchan * nsamp, D, nout,
                                                                                    tb, (unsigned)runs, d_out);
    return af_cuda_check(cudaGetLastError(), "af_downsample launch");
} catch (...) {
    return af_host_exception("af_downsample");
}

// ---------------------------------------------------------------- zero-DM
// Zero-DM filter: q[t] = round_half_up(sum_c X[c][t] / nchan), out = clip(X - q + 128).
// Up to 4096 channels, a cluster of 1, 2, 4 or 8 blocks owns a tile of 128
// samples of every channel and holds it in shared memory, so that the input is
// read once (k_zerodm_tile).  More channels, and long rows of few (whose tiles would
// leave most of a block idle): a block owns 512 samples of every channel and
// reads them twice (k_zerodm16: rows of whole 16-byte pieces), or one thread per 4
// samples (k_zerodm, any shape).
// In place is safe: a tile's samples are read before any of them is written,
// and only its own bytes are written.
namespace {

constexpr int kZW = 16;           // warps per block (channel split)
constexpr int kZTile = 512;       // two-read kernel: samples per block
constexpr int kZT = 128;          // generic kernel: threads per block
constexpr int kZS = 128;          // held tile: samples (8 lanes of 16 bytes per channel)
constexpr int kZV = 8;            // held tile: 16-byte pieces per thread
constexpr int kZC = 4 * kZW * kZV;  // held tile: channels per block (512)
constexpr int kZPieces = kZV * kZW * 32;                     // held pieces of a block (64 KB) ...
constexpr int kZSmemA = 16 * kZPieces, kZSmemU = kZSmemA + 16 * kZC;  // ... and a ninth per channel off a boundary

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// Bytes k .. k + 15 of the 32 bytes a, b (0 <= k < 16).
__device__ __forceinline__ uint4 window16(const uint4& a, const uint4& b, int k)
{
    const bool s8 = (k & 8) != 0, s4 = (k & 4) != 0;
    const uint32_t t0 = s8 ? a.z : a.x, t1 = s8 ? a.w : a.y, t2 = s8 ? b.x : a.z, t3 = s8 ? b.y : a.w,
                   t4 = s8 ? b.z : b.x, t5 = s8 ? b.w : b.y;
    const uint32_t u0 = s4 ? t1 : t0, u1 = s4 ? t2 : t1, u2 = s4 ? t3 : t2, u3 = s4 ? t4 : t3, u4 = s4 ? t5 : t4;
    const uint32_t sh = 8u * (uint32_t)(k & 3);
    return make_uint4(__funnelshift_r(u0, u1, sh), __funnelshift_r(u1, u2, sh), __funnelshift_r(u2, u3, sh),
                      __funnelshift_r(u3, u4, sh));
}

__device__ __forceinline__ uint32_t byte_of(const uint4& v, int i)
{
    const uint32_t w = i < 8 ? (i < 4 ? v.x : v.y) : (i < 12 ? v.z : v.w);
    return (w >> (8 * (i & 3))) & 0xFFu;
}

// Lane l of 8 owns samples 16 l .. 16 l + 15 of a channel's tile; a warp takes
// 4 channels per step, a block 64, up to kZV steps.  The pieces arrive by
// 16-byte asynchronous copies, so a block holds its 64 KB without registers and
// three blocks an SM overlap their reads, reductions and writes.  16-bit lane
// sums over a warp's channels (at most 32 x 255), 32-bit across warps in shared
// memory and across the cluster through distributed shared memory.  ALIGNED:
// every row starts on a 16-byte boundary and is whole 16-byte pieces.
// Otherwise a channel's samples lie in nine aligned pieces; a lane cuts its 16
// bytes out of two of them, and stores the aligned piece that its first and
// lane l - 1's last bytes form; only a tile's two ends go byte by byte.
// Bound by HBM and by the latency of a tile's chain (copy, two reductions, a
// cluster barrier, store).  4096 x 2^18: 0.61 ms with two reads (3.2 GB moved),
// 0.37 ms so; held in registers, two blocks an SM, 0.52 ms.  Rows off a 16-byte
// boundary (2064 x 77251): 2.58 ms byte by byte, 0.27 ms so.
template <bool ALIGNED>
__global__ void __launch_bounds__(kZW * 32, ALIGNED ? 3 : 2)
k_zerodm_tile(const uint8_t* X, int nchan, int64_t nsamp, uint8_t* out)
{
    extern __shared__ __align__(16) uint4 held[];          // [kZV][block's threads], then the ninth pieces
    __shared__ __align__(16) uint32_t part[kZW][kZS / 2];  // per warp: 16-bit sums, as the registers hold them
    __shared__ uint32_t sum[kZS];                          // this block's channel sums
    __shared__ __align__(16) uint16_t nq[kZS];             // 128 - mean, in the registers' order
    cg::cluster_group cluster = cg::this_cluster();
    const int parts = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, l = lane & 7;
    const int64_t t0 = (int64_t)(blockIdx.x / parts) * kZS;
    const int per = (nchan + parts - 1) / parts;
    const int c0 = rank * per + 4 * warp + (lane >> 3), c1 = min(nchan, (rank + 1) * per);
    const int64_t step = (int64_t)(4 * kZW) * nsamp;  // bytes between a lane's channels
    const int64_t at0 = (int64_t)c0 * nsamp + t0 + 16 * l;
    const int nval = (int)min((int64_t)kZS, nsamp - t0);    // the tile's samples
    const int nb = max(0, min(16, nval - 16 * l));          // the lane's
    const int nv = c0 < c1 ? (c1 - c0 + 4 * kZW - 1) / (4 * kZW) : 0;  // the lane's channels
    uint4* ninth = held + kZPieces + 4 * warp + (lane >> 3);           // of step i: + 4 kZW i

    // 1. the copies
    {
        const uint8_t* a = X + at0;
        const uint8_t* const xend = X + (int64_t)nchan * nsamp;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(held + tid);
#pragma unroll
        for (int i = 0; i < kZV; i++, a += step) {
            if (i >= nv) break;
            if (ALIGNED) {
                if (nb > 0) cp_async16(dst + i * (16 * kZW * 32), a);
            } else {
                const int m = (int)(reinterpret_cast<uintptr_t>(a) & 15);  // the same in a channel's 8 lanes
                // a piece that reaches past the input is copied byte by byte
                auto fetch = [&](const uint8_t* src, uint4* to) {
                    if (src >= X && src + 16 <= xend) {
                        cp_async16((uint32_t)__cvta_generic_to_shared(to), src);
                    } else {
                        for (int j = 0; j < 16; j++)
                            reinterpret_cast<uint8_t*>(to)[j] = src + j >= X && src + j < xend ? src[j] : (uint8_t)0;
                    }
                };
                if (16 * l - m < nval) fetch(a - m, held + i * (kZW * 32) + tid);
                if (l == 7 && m > 0 && kZS - m < nval) fetch(a - m + 16, ninth + 4 * kZW * i);
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (!ALIGNED) __syncwarp();  // a lane reads its neighbour's piece
    }
    // the lane's 16 samples of step i
    auto mine = [&](int i) -> uint4 {
        const uint4 p = held[i * (kZW * 32) + tid];
        if (ALIGNED) return p;
        const int m = (int)((reinterpret_cast<uintptr_t>(X) + (uintptr_t)(at0 + i * step)) & 15);
        if (m == 0) return p;
        return window16(p, l == 7 ? ninth[4 * kZW * i] : held[i * (kZW * 32) + tid + 1], m);
    };

    // 2. sums over the block's channels
    uint32_t s[8];  // word j of the 16 bytes: s[2 j] = bytes 0, 2, s[2 j + 1] = bytes 1, 3
#pragma unroll
    for (int j = 0; j < 8; j++) s[j] = 0u;
    if (nb > 0)
        for (int i = 0; i < nv; i++) {
            const uint4 v = mine(i);
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < 4; j++) {
                s[2 * j] += w[j] & 0x00FF00FFu;
                s[2 * j + 1] += __byte_perm(w[j], 0u, 0x4341);
            }
        }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 8; j++) {
        s[j] += __shfl_xor_sync(0xffffffffu, s[j], 8);
        s[j] += __shfl_xor_sync(0xffffffffu, s[j], 16);
    }
    if (lane < 8) {
        *reinterpret_cast<uint4*>(&part[warp][8 * lane]) = make_uint4(s[0], s[1], s[2], s[3]);
        *reinterpret_cast<uint4*>(&part[warp][8 * lane + 4]) = make_uint4(s[4], s[5], s[6], s[7]);
    }
    __syncthreads();
    uint32_t t = 0;
    if (tid < kZS) {  // thread h: half h & 1 of word h >> 1
#pragma unroll
        for (int w = 0; w < kZW; w++) t += reinterpret_cast<const uint16_t*>(part[w])[tid];
        sum[tid] = t;
    }
    // 3. the mean, from every block's sums
    if (parts > 1) {
        cluster.sync();
        if (tid < kZS) {
            t = 0;
            for (int r = 0; r < parts; r++) t += *cluster.map_shared_rank(&sum[tid], r);
        }
    }
    if (tid < kZS) nq[tid] = (uint16_t)(int16_t)(128 - (int)((2u * t + (uint32_t)nchan) / (2u * (uint32_t)nchan)));
    __syncthreads();
    // arrives here, waits at the end: no block leaves while another may still read its sums
    if (parts > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    uint32_t d[8];
    {
        const uint4 a = *reinterpret_cast<const uint4*>(&nq[16 * l]), b = *reinterpret_cast<const uint4*>(&nq[16 * l + 8]);
        d[0] = a.x, d[1] = a.y, d[2] = a.z, d[3] = a.w, d[4] = b.x, d[5] = b.y, d[6] = b.z, d[7] = b.w;
    }
    // 4. the filtered samples; off a boundary, every lane of a warp runs every step (shuffles)
    const int steps = ALIGNED ? (nb > 0 ? nv : 0) : kZV;
    uint8_t* o = out + at0;
    for (int i = 0; i < steps; i++, o += step) {
        const bool live = i < nv && nb > 0;
        const uint4 v = ALIGNED || live ? mine(i) : make_uint4(0u, 0u, 0u, 0u);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        uint32_t r[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {  // max(0, min(255, x + 128 - q)), two samples at a time
            const uint32_t e = __viaddmin_s16x2_relu(w[j] & 0x00FF00FFu, d[2 * j], 0x00FF00FFu);
            const uint32_t f = __viaddmin_s16x2_relu(__byte_perm(w[j], 0u, 0x4341), d[2 * j + 1], 0x00FF00FFu);
            r[j] = e | f << 8;
        }
        const uint4 own = make_uint4(r[0], r[1], r[2], r[3]);
        if (ALIGNED) {
            *reinterpret_cast<uint4*>(o) = own;
        } else {
            uint4 prev;
            prev.x = __shfl_up_sync(0xffffffffu, own.x, 1);
            prev.y = __shfl_up_sync(0xffffffffu, own.y, 1);
            prev.z = __shfl_up_sync(0xffffffffu, own.z, 1);
            prev.w = __shfl_up_sync(0xffffffffu, own.w, 1);
            if (live) {
                const int m = (int)(reinterpret_cast<uintptr_t>(o) & 15);  // the same in a channel's 8 lanes
                const int first = 16 - m;  // own bytes in the aligned piece at o - m; lane l - 1's last m precede them
                if (m == 0 && nb == 16) {
                    *reinterpret_cast<uint4*>(o) = own;
                } else {
                    if (l > 0 && m > 0 && nb >= first) {
                        *reinterpret_cast<uint4*>(o - m) = window16(prev, own, first);
                    } else {
                        for (int j = 0; j < min(first, nb); j++) o[j] = (uint8_t)byte_of(own, j);
                        if (l > 0 && m > 0)
                            for (int j = first; j < 16; j++) o[j - 16] = (uint8_t)byte_of(prev, j);
                    }
                    // own last m bytes are the next lane's to store, unless there is none
                    if (l == 7 || nval - 16 * (l + 1) <= 0)
                        for (int j = first; j < nb; j++) o[j] = (uint8_t)byte_of(own, j);
                }
            }
            __syncwarp();
        }
    }
    __syncwarp();  // lanes past the row or its channels ran fewer steps
    if (parts > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__global__ void __launch_bounds__(kZW * 32)
k_zerodm16(const uint8_t* X, int nchan, int64_t nsamp, uint8_t* out)
{
    __shared__ uint32_t part[kZW][kZTile];
    __shared__ int32_t q[kZTile];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t t0 = (int64_t)blockIdx.x * kZTile + 16 * lane;
    const int c0 = (int)((int64_t)nchan * warp / kZW);
    // the lane's 16 samples are in the row, or all past it: no channels then
    const int c1 = t0 < nsamp ? (int)((int64_t)nchan * (warp + 1) / kZW) : c0;
    uint32_t sum[16];
#pragma unroll
    for (int i = 0; i < 16; i++) sum[i] = 0u;
    for (int cb = c0; cb < c1; cb += 256) {
        const int ce = min(c1, cb + 256);
        uint32_t E[4] = {0u, 0u, 0u, 0u}, O[4] = {0u, 0u, 0u, 0u};
#pragma unroll 4
        for (int c = cb; c < ce; c++) {
            const uint4 v = *reinterpret_cast<const uint4*>(X + (int64_t)c * nsamp + t0);
            const uint32_t wv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < 4; j++) {
                E[j] += wv[j] & 0x00FF00FFu;
                O[j] += __byte_perm(wv[j], 0u, 0x4341);
            }
        }
#pragma unroll
        for (int j = 0; j < 4; j++) {
            sum[4 * j + 0] += E[j] & 0xFFFFu;
            sum[4 * j + 1] += O[j] & 0xFFFFu;
            sum[4 * j + 2] += E[j] >> 16;
            sum[4 * j + 3] += O[j] >> 16;
        }
    }
#pragma unroll
    for (int i = 0; i < 16; i++) part[warp][16 * lane + i] = sum[i];
    __syncthreads();
    for (int i = threadIdx.x; i < kZTile; i += kZW * 32) {
        uint32_t s = 0;
#pragma unroll
        for (int w = 0; w < kZW; w++) s += part[w][i];
        q[i] = (int32_t)((2u * s + (uint32_t)nchan) / (2u * (uint32_t)nchan)) - 128;
    }
    __syncthreads();
    int32_t qq[16];
#pragma unroll
    for (int i = 0; i < 16; i++) qq[i] = q[16 * lane + i];
#pragma unroll 4
    for (int c = c0; c < c1; c++) {
        const int64_t o = (int64_t)c * nsamp + t0;
        const uint4 v = *reinterpret_cast<const uint4*>(X + o);  // plain load: X may alias out
        const uint32_t wv[4] = {v.x, v.y, v.z, v.w};
        uint32_t r[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            uint32_t acc = 0;
#pragma unroll
            for (int b = 0; b < 4; b++) {
                const int x = (int)((wv[j] >> (8 * b)) & 0xFFu) - qq[4 * j + b];
                acc |= (uint32_t)min(255, max(0, x)) << (8 * b);
            }
            r[j] = acc;
        }
        *reinterpret_cast<uint4*>(out + o) = make_uint4(r[0], r[1], r[2], r[3]);
    }
}

__global__ void __launch_bounds__(kZT)
k_zerodm(const uint8_t* X, int nchan, int64_t nsamp, uint8_t* out)
{
    const int64_t t = ((int64_t)blockIdx.x * kZT + threadIdx.x) * 4;
    if (t >= nsamp) return;
    const int n = (int)min((int64_t)4, nsamp - t);
    uint32_t s[4] = {0u, 0u, 0u, 0u};
    for (int c = 0; c < nchan; c++)
        for (int i = 0; i < n; i++) s[i] += X[(int64_t)c * nsamp + t + i];
    int q[4];
#pragma unroll
    for (int i = 0; i < 4; i++) q[i] = (int)((2u * s[i] + (uint32_t)nchan) / (2u * (uint32_t)nchan)) - 128;
    for (int c = 0; c < nchan; c++)
        for (int i = 0; i < n; i++) {
            const int64_t o = (int64_t)c * nsamp + t + i;
            const int v = (int)X[o] - q[i];
            out[o] = (uint8_t)min(255, max(0, v));
        }
}

}  // namespace

extern "C" int af_zerodm(const uint8_t* d_in, int nchan, int64_t nsamp, uint8_t* d_out, void* stream)
try {
    if (!d_in || !d_out) return af_set_error(AF_EINVAL, "af_zerodm: NULL buffer");
    if (nchan < 1 || nchan > 65536 || nsamp < 1) return af_set_error(AF_EINVAL, "af_zerodm: bad shape");
    cudaStream_t s = (cudaStream_t)stream;
    const bool aligned = nsamp % 16 == 0 && ((uintptr_t)d_in % 16 == 0) && ((uintptr_t)d_out % 16 == 0);
    // Blocks per tile: the fewest that hold every channel.  Long rows of few channels go to the kernels that read twice.  Tile /
    // those, us: 1 x 2^24 aligned 385 / 31, off a boundary 1328 / 31; 16 x 2^24 523 / 373 and 1866 / 302; 64 x 2^23 354 / 298 and
    // 1253 / 725; 96 x 2^22 174 / 189; 128 x 2^22 236 / 244 and 923 / 823; 256 x 2^21 178 / 237 and 742 / 857; 64 x 2^14 4.2 / 6.2 and 6.2 / 47.
    int parts = 1;
    while (parts * kZC < nchan) parts *= 2;
    const int64_t tiles = (nsamp + kZS - 1) / kZS;
    // (k_zerodm16 wants a channel for each of its warps.)
    const bool few = nchan <= 2 ||
                     (aligned ? nchan < 72 && nsamp >= (nchan < kZW ? std::max(65536, 16384 * nchan) : 65536)
                              : nchan < 160 && nsamp >= 4096 * (int64_t)nchan);
    if (nchan <= 8 * kZC && !few && tiles * parts <= 0x7fffffff) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(tiles * parts));
        cfg.blockDim = dim3(kZW * 32);
        cfg.stream = s;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)parts;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        cfg.dynamicSmemBytes = aligned ? kZSmemA : kZSmemU;
        if (int rc = af_ensure_smem(aligned ? (const void*)k_zerodm_tile<true> : (const void*)k_zerodm_tile<false>,
                                    cfg.dynamicSmemBytes))
            return rc;
        return af_cuda_check(aligned ? cudaLaunchKernelEx(&cfg, k_zerodm_tile<true>, d_in, nchan, nsamp, d_out)
                                     : cudaLaunchKernelEx(&cfg, k_zerodm_tile<false>, d_in, nchan, nsamp, d_out),
                             "af_zerodm launch");
    }
    if (aligned && nchan >= kZW) {
        const int64_t blocks = (nsamp + kZTile - 1) / kZTile;
        if (blocks > 0x7fffffff) return af_set_error(AF_EINVAL, "af_zerodm: input too large");
        k_zerodm16<<<(unsigned)blocks, kZW * 32, 0, s>>>(d_in, nchan, nsamp, d_out);
    } else {
        const int64_t blocks = (nsamp + 4 * kZT - 1) / (4 * kZT);
        if (blocks > 0x7fffffff) return af_set_error(AF_EINVAL, "af_zerodm: input too large");
        k_zerodm<<<(unsigned)blocks, kZT, 0, s>>>(d_in, nchan, nsamp, d_out);
    }
    return af_cuda_check(cudaGetLastError(), "af_zerodm launch");
} catch (...) {
    return af_host_exception("af_zerodm");
}
