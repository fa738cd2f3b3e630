// snr.cu -- boxcar matched filter and S/N normalisation (step (iii) of the
// single-pulse workflow, Sec. 1 of the paper; definitions as in afgb.h).
//
//   B_w[t]  = sum_{k=t}^{t+w-1} Y[d][k]
//   snr_w   = (nout*B_w - w*S) / (nout*sigma*sqrt(w))
//           = (B_w - q_w) * k_w - c_w,   q_w = floor(w*S/nout),
//             k_w = 1/(sigma*sqrt(w)),  c_w = ((w*S - q_w*nout)/nout) * k_w
//
// The split keeps the cancellation B_w - w*mu exact in integers: (B_w - q_w)
// is an exact integer and only the final scale is rounded, so the float
// result is within a few ulp of the exact S/N.  Window sums come from 32-bit
// prefix sums taken modulo 2^32, which are exact as long as every window sum
// is below 2^32 (checked on the host: w * 255 * nchan < 2^32).
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "internal.h"

namespace cg = cooperative_groups;

namespace {

__device__ __forceinline__ double i128_to_double(__int128 v)
{
    const bool neg = v < 0;
    const unsigned __int128 u = neg ? (unsigned __int128)(-v) : (unsigned __int128)v;
    const double r = (double)(uint64_t)(u >> 64) * 18446744073709551616.0 + (double)(uint64_t)u;
    return neg ? -r : r;
}

// One thread per (row, width): the constants q, k, c above, from the exact
// row sums.  sigma^2 = (nout*Q - S^2)/nout^2 with the numerator in 128 bits.
__global__ void k_rowconst(const af_rowstats_t* __restrict__ st, int ndm, int64_t nout, af_widths_t w,
                           af_rowconst_t* __restrict__ rc)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ndm * w.n) return;
    const int d = i / w.n, wi = i % w.n;
    const int64_t S = st[d].sum, Q = st[d].sumsq;
    const __int128 vnum = (__int128)nout * Q - (__int128)S * S;
    const double var = i128_to_double(vnum) / ((double)nout * (double)nout);
    const double sigma = var > 0.0 ? sqrt(var) : 0.0;
    const int64_t W = w.w[wi];
    const int64_t ws = W * S;            // < nout * 2^32 <= 2^63 by the width check
    const int64_t q = ws / nout;         // S >= 0: truncation is the floor
    const int64_t r = ws - q * nout;     // 0 <= r < nout
    af_rowconst_t o;
    o.q = q;
    if (sigma > 0.0) {
        const double k = 1.0 / (sigma * sqrt((double)W));
        o.k = (float)k;
        o.c = (float)(((double)r / (double)nout) * k);
    } else {
        o.k = 0.0f;
        o.c = 0.0f;
    }
    rc[(int64_t)d * AF_MAX_WIDTHS + wi] = o;
}

constexpr int kBT = 256;             // threads per block
constexpr int kBW = kBT / 32;        // warps
constexpr int kFloatBits = 22;       // the float path needs |prefix| and |q - w mu0| below 2^22

// Two fp32 operations in one instruction (each rounded like the scalar one).
__device__ __forceinline__ uint64_t pack2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// One width of a tile's outputs, e = q - w mu0 (an integer, or -e as a float
// where the float path runs) and the constants twice, as the paired
// instructions take them.
struct __align__(16) BoxWidth {
    int32_t e, e2;
    float k, k2;
    float nc, nc2;   // -c
    int w, pad;
};

__device__ __forceinline__ float max3(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

enum { kPathFloat, kPathInt, kPathWide };

// Pairs of prefix words P[i + w] .. P[i + w + 3] for i % 4 == 0, given the
// four words at i (x) and at i + 4 (y), r = w % 4.
__device__ __forceinline__ void shift_words(const ulonglong2& x, const ulonglong2& y, int r, uint64_t (&p)[2])
{
    if (r == 1) {
        p[0] = x.x >> 32 | x.y << 32;
        p[1] = x.y >> 32 | y.x << 32;
    } else if (r == 2) {
        p[0] = x.y;
        p[1] = y.x;
    } else {
        p[0] = x.y >> 32 | y.x << 32;
        p[1] = y.x >> 32 | y.y << 32;
    }
}

// Every width's S/N of the four outputs lt .. lt + 3 (lt % 4 == 0): the best
// and its index.  PATH kPathFloat: the words are floats holding exact integers
// below 2^22, so both differences are exact in fp32 and equal the converted
// integer difference bit for bit; kPathInt: 32-bit integers; kPathWide: 32-bit
// prefix, 64-bit difference.  TAIL: windows that pass the row's end do not
// count.  Widths are taken three at a time (the list padded with copies of its
// last, which never win a tie against it): one three-input maximum, one
// comparison with the best so far, and the first two values of the winning
// group kept; which of its three widths it was is found once, at the end.
template <int PATH, bool TAIL>
__device__ __forceinline__ void box_outputs(const uint32_t* P, const BoxWidth* sw, const int64_t* sq, int nw, int left,
                                            int lt, float (&best)[4], int (&bi)[4])
{
    const ulonglong2 p0 = *reinterpret_cast<const ulonglong2*>(P + lt);
    float s0[4], s1[4];
    const uint64_t minus1 = pack2(-1.0f, -1.0f);
    auto group = [&](int k0, auto first) {
        float v[3][4];
#pragma unroll
        for (int i = 0; i < 3; i++) {
            const BoxWidth c = sw[k0 + i];
            const uint32_t* Pw = P + lt + (c.w & ~3);
            const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(Pw);
            uint64_t p[2] = {x.x, x.y};
            if (c.w & 3) shift_words(x, *reinterpret_cast<const ulonglong2*>(Pw + 4), c.w & 3, p);  // uniform
            if (PATH == kPathFloat) {
                const uint64_t ne = pack2(__int_as_float(c.e), __int_as_float(c.e2));
                const uint64_t k2 = pack2(c.k, c.k2), nc = pack2(c.nc, c.nc2);
                unpack2(fma2(add2(fma2(p0.x, minus1, p[0]), ne), k2, nc), v[i][0], v[i][1]);
                unpack2(fma2(add2(fma2(p0.y, minus1, p[1]), ne), k2, nc), v[i][2], v[i][3]);
            } else {
                const int64_t qq = PATH == kPathWide ? sq[k0 + i] : 0;
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const uint64_t own = j < 2 ? p0.x : p0.y;
                    const uint32_t B = (uint32_t)(p[j >> 1] >> (32 * (j & 1))) - (uint32_t)(own >> (32 * (j & 1)));
                    const float x1 = PATH == kPathInt ? (float)(int32_t)(B - (uint32_t)c.e) : (float)((int64_t)B - qq);
                    v[i][j] = fmaf(x1, c.k, c.nc);
                }
            }
            if (TAIL) {
#pragma unroll
                for (int j = 0; j < 4; j++)
                    if (lt + j + c.w > left) v[i][j] = -INFINITY;
            }
        }
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const float m = max3(v[0][j], v[1][j], v[2][j]);
            if (decltype(first)::value) {
                best[j] = m;
                s0[j] = v[0][j];
                s1[j] = v[1][j];
                bi[j] = 0;
            } else if (m > best[j]) {
                best[j] = m;
                s0[j] = v[0][j];
                s1[j] = v[1][j];
                bi[j] = k0;
            }
        }
    };
    group(0, std::true_type{});
    for (int k0 = 3; k0 < nw; k0 += 3) group(k0, std::false_type{});
#pragma unroll
    for (int j = 0; j < 4; j++) {
        bi[j] += s0[j] == best[j] ? 0 : (s1[j] == best[j] ? 1 : 2);
        if (TAIL && best[j] == -INFINITY) bi[j] = AF_NO_WIDTH;
    }
}

// Block = one tile of one row: `outs` outputs from t0 on, and the prefix words
// of the tile and its halo, kBW * NCH chunks of 128; t0 is a multiple of outs
// less the row's misalignment (0 to 3 words), so that every load and store is
// a whole 16-byte one wherever the row starts (rows of odd length: three of
// four start off a 16-byte boundary).
//  1. NCH consecutive chunks per warp are read, one 16-byte load per lane, all
//     issued first; values outside the row count as mu0, an integer near the
//     row's mean.
//  2. P[j] = sum_{k<j} (Y[t0+k] - mu0) mod 2^32: 4 values per lane, a warp
//     scan per chunk, chunk and warp offsets; one 16-byte store per lane.  The
//     window sum is P[t+w] - P[t] + w mu0, and B - q = P[t+w] - P[t] - e with
//     e = q - w mu0.
//  3. If no |P| of the tile reaches 2^22 (noise: a random walk of a few tens of
//     thousands), P is stored as floats: B - q then takes two exact fp32
//     operations, issued two outputs at a time, and no integer-to-float
//     conversion per (output, width).  Otherwise the integers are stored.
//  4. A thread takes 4 consecutive outputs at a time, so one 16-byte shared load
//     brings P[t+w] for four outputs.
// Bound by instruction issue (99 warp instructions per 32 outputs at 9 widths:
// 38 of them loads, scan and stores, then 20 per three widths).  1001 x 215261
// plane, 9 widths up to 256: 0.86 ms with an integer difference, a conversion
// and a 4-byte shared load per (output, width) and 4-byte global loads on rows
// off a 16-byte boundary; 0.68 ms so.  Measured slower: two 4-output groups per
// thread together (80 registers, spills: 0.80 ms), one comparison and two
// selects per width (0.75 ms), 3 or 5 blocks per SM (0.73 ms).
template <bool SMALL, int NCH>
__global__ void __launch_bounds__(kBT, NCH <= 6 ? 4 : 3)
k_boxcar(const int32_t* __restrict__ Y, int ndm, int64_t nout, int outs, af_widths_t w,
         const af_rowconst_t* __restrict__ rc, float* __restrict__ snr, uint8_t* __restrict__ bw)
{
    constexpr int kWords = kBW * NCH * 128;
    __shared__ __align__(16) uint32_t P[kWords + 8];
    __shared__ BoxWidth sw[AF_MAX_WIDTHS + 2];
    __shared__ int64_t sq[AF_MAX_WIDTHS + 2];
    __shared__ __align__(16) uint32_t swarp[kBW];

    const int64_t d = blockIdx.y + (int64_t)gridDim.y * blockIdx.z;
    if (d >= ndm) return;
    const int nw = w.n;
    const int nw3 = (nw + 2) / 3 * 3;  // the list in whole groups of three
    const int32_t* row = Y + d * nout;
    const int mis = (int)((reinterpret_cast<uintptr_t>(row) >> 2) & 3);
    const int64_t t0 = (int64_t)blockIdx.x * outs - mis;
    if (t0 >= nout) return;
    const int first = blockIdx.x == 0 ? mis : 0;                                 // words before the row's start
    const int left = (int)(nout - t0 < 2 * kWords ? nout - t0 : 2 * kWords);     // row samples from t0 on (clipped)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const af_rowconst_t* rcd = rc + d * AF_MAX_WIDTHS;

    // 1. loads
    const int32_t* yt = row + t0;
    const int i0 = warp * NCH * 128 + 4 * lane;
    int4 v[NCH];
#pragma unroll
    for (int u = 0; u < NCH; u++) {
        const int i = i0 + 128 * u;
        v[u] = make_int4(0, 0, 0, 0);
        if (i >= first && i + 3 < left) v[u] = __ldg(reinterpret_cast<const int4*>(yt + i));
    }
    const int32_t mu0 = SMALL ? __float2int_rn(__fdividef(__ll2float_rn(rcd[nw - 1].q), (float)w.w[nw - 1])) : 0;
    bool wide_e = false;  // an offset e too large for the float path
    if (tid < nw3) {
        const int k = min(tid, nw - 1);
        const af_rowconst_t c = rcd[k];
        BoxWidth o;
        o.w = w.w[k];
        const int32_t e = (int32_t)((uint32_t)c.q - (uint32_t)o.w * (uint32_t)mu0);
        wide_e = e <= -(1 << kFloatBits) || e >= (1 << kFloatBits);
        o.e = o.e2 = e;
        o.k = o.k2 = c.k;
        o.nc = o.nc2 = -c.c;
        o.pad = 0;
        sw[tid] = o;
        sq[tid] = c.q;
    }
#pragma unroll
    for (int u = 0; u < NCH; u++) {
        const int i = i0 + 128 * u;
        if (i >= first && i + 3 < left) {
            v[u].x -= mu0;
            v[u].y -= mu0;
            v[u].z -= mu0;
            v[u].w -= mu0;
        } else if (i + 3 >= first && i < left) {  // the row's ends
            if (i >= first) v[u].x = __ldg(yt + i) - mu0;
            if (i + 1 >= first && i + 1 < left) v[u].y = __ldg(yt + i + 1) - mu0;
            if (i + 2 >= first && i + 2 < left) v[u].z = __ldg(yt + i + 2) - mu0;
            if (i + 3 < left) v[u].w = __ldg(yt + i + 3) - mu0;
        }
    }

    // 2. exclusive prefix sums: ex[u] = sum of everything of the warp before the lane's chunk-u values
    uint32_t ex[NCH], run = 0;
#pragma unroll
    for (int u = 0; u < NCH; u++) {
        const uint32_t own = (uint32_t)v[u].x + (uint32_t)v[u].y + (uint32_t)v[u].z + (uint32_t)v[u].w;
        uint32_t incl = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        ex[u] = run + incl - own;
        run += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) swarp[warp] = run;
    __syncthreads();
    uint32_t off = 0;
#pragma unroll
    for (int k = 0; k < kBW; k++) off += k < warp ? swarp[k] : 0u;
    int32_t hi = 0, lo = 0;  // range of the tile's prefix sums
#pragma unroll
    for (int u = 0; u < NCH; u++) {  // v[u] becomes the lane's four prefix words
        const uint32_t a = off + ex[u], b = a + (uint32_t)v[u].x, c = b + (uint32_t)v[u].y, e = c + (uint32_t)v[u].z;
        v[u] = make_int4((int)a, (int)b, (int)c, (int)e);
        hi = __vimax3_s32(__vimax3_s32(hi, v[u].x, v[u].y), v[u].z, v[u].w);
        lo = __vimin3_s32(__vimin3_s32(lo, v[u].x, v[u].y), v[u].z, v[u].w);
    }
    const bool bad = wide_e || hi >= (1 << kFloatBits) || lo <= -(1 << kFloatBits);
    // 3. the prefix words in the form the tile's path reads
    const bool flt = SMALL && __syncthreads_or(bad) == 0;
#pragma unroll
    for (int u = 0; u < NCH; u++) {
        if (flt)
            *reinterpret_cast<float4*>(P + i0 + 128 * u) =
                make_float4((float)v[u].x, (float)v[u].y, (float)v[u].z, (float)v[u].w);
        else
            *reinterpret_cast<int4*>(P + i0 + 128 * u) = v[u];
    }
    if (flt && tid < nw3) sw[tid].e = sw[tid].e2 = __float_as_int(-(float)sw[tid].e);
    __syncthreads();

    // 4. every width's S/N and the best
    const int nown = min(outs, left);                     // the tile's outputs
    const bool tail = left < outs + w.w[nw - 1];          // some windows pass the row's end (uniform)
    float* so = snr + d * nout + t0;
    uint8_t* bo = bw ? bw + d * nout + t0 : nullptr;
    const bool vec = (reinterpret_cast<uintptr_t>(so) & 15) == 0 && (reinterpret_cast<uintptr_t>(bo) & 3) == 0;
#pragma unroll 1
    for (int lt = 4 * tid; lt < nown; lt += 4 * kBT) {
        float best[4];
        int bi[4];
        if (!SMALL) {
            if (tail) box_outputs<kPathWide, true>(P, sw, sq, nw, left, lt, best, bi);
            else box_outputs<kPathWide, false>(P, sw, sq, nw, left, lt, best, bi);
        } else if (flt) {
            if (tail) box_outputs<kPathFloat, true>(P, sw, sq, nw, left, lt, best, bi);
            else box_outputs<kPathFloat, false>(P, sw, sq, nw, left, lt, best, bi);
        } else {
            if (tail) box_outputs<kPathInt, true>(P, sw, sq, nw, left, lt, best, bi);
            else box_outputs<kPathInt, false>(P, sw, sq, nw, left, lt, best, bi);
        }
        if (vec && lt >= first && lt + 3 < nown) {
            *reinterpret_cast<float4*>(so + lt) = make_float4(best[0], best[1], best[2], best[3]);
            if (bo)
                *reinterpret_cast<uint32_t*>(bo + lt) =
                    (uint32_t)bi[0] | (uint32_t)bi[1] << 8 | (uint32_t)bi[2] << 16 | (uint32_t)bi[3] << 24;
        } else {
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (lt + j >= first && lt + j < nown) {
                    so[lt + j] = best[j];
                    if (bo) bo[lt + j] = (uint8_t)bi[j];
                }
        }
    }
}

template <bool SMALL, int NCH>
int launch_boxcar_nch(const int32_t* d_plane, int ndm, int64_t nout, const af_widths_t& w,
                      const af_rowconst_t* d_rowconst, float* d_best_snr, uint8_t* d_best_w, cudaStream_t s)
{
    // a tile's prefix words less its halo, in whole 16-byte groups
    const int outs = (kBW * NCH * 128 - w.w[w.n - 1]) & ~3;
    const int64_t tiles = (nout + 3 + outs - 1) / outs;  // a row may start up to 3 words into its first tile
    if ((long double)tiles * ndm > 0x7fffffffLL) return af_set_error(AF_EINVAL, "boxcar: problem too large for one grid");
    const int gy = ndm < 32768 ? ndm : 32768;
    const dim3 grid((unsigned)tiles, (unsigned)gy, (unsigned)((ndm + gy - 1) / gy));
    k_boxcar<SMALL, NCH><<<grid, kBT, 0, s>>>(d_plane, ndm, nout, outs, w, d_rowconst, d_best_snr, d_best_w);
    return af_cuda_check(cudaGetLastError(), "boxcar launch");
}

int launch_boxcar_tiles(const int32_t* d_plane, int ndm, int64_t nout, const af_widths_t& w,
                        const af_rowconst_t* d_rowconst, float* d_best_snr, uint8_t* d_best_w, cudaStream_t s)
{
    // 6144 prefix words per tile for widths up to 1024 samples, 12288 up to 8192; 2048 for widths up to 512 of planes whose
    // larger tiles are no more than the four blocks that each SM holds (a block then works through six steps while
    // others are idle).  32 widths up to 32, us by 6144 / 2048: 64 x 5000 28.8 / 20.7, 1 x 10^6 32.9 / 24.8, 200 x 12,000 (600 tiles)
    // 51.3 / 41.1, 500 x 28,000 (2500) 172.8 / 168.0; 5 widths up to 256: 300 x 6000 21.2 / 16.7, 100 x 40,000 (700) 21.2 / 23.0,
    // 500 x 28,000 49.2 / 57.4.
    int dev = 0, nsm = 0;
    AF_CUDA(cudaGetDevice(&dev));
    AF_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    const int wmax = w.w[w.n - 1];
    const bool near = wmax <= 1024;
    const int64_t outs = kBW * 6 * 128 - wmax;  // outputs of a 6144-word tile
    const bool few = wmax <= 512 && (nout + outs - 1) / outs * ndm <= 4 * (int64_t)nsm;
    if (few)
        return w.small ? launch_boxcar_nch<true, 2>(d_plane, ndm, nout, w, d_rowconst, d_best_snr, d_best_w, s)
                       : launch_boxcar_nch<false, 2>(d_plane, ndm, nout, w, d_rowconst, d_best_snr, d_best_w, s);
    if (w.small)
        return near ? launch_boxcar_nch<true, 6>(d_plane, ndm, nout, w, d_rowconst, d_best_snr, d_best_w, s)
                    : launch_boxcar_nch<true, 12>(d_plane, ndm, nout, w, d_rowconst, d_best_snr, d_best_w, s);
    return near ? launch_boxcar_nch<false, 6>(d_plane, ndm, nout, w, d_rowconst, d_best_snr, d_best_w, s)
                : launch_boxcar_nch<false, 12>(d_plane, ndm, nout, w, d_rowconst, d_best_snr, d_best_w, s);
}

// ---------------------------------------------------------------- robust S/N
// Per-row median and MAD (lower medians, exact) by radix selection: one block
// per row; each pass histograms a window of the value range into at most 2048
// bins in shared memory and keeps the bin holding the wanted rank, so a window
// of R values takes ceil(log2(R) / 11) passes.
//
// Windows.  A first pass takes the row's minimum, maximum, mean mu and a bound
// s >= sigma on its standard deviation.  Any median m of a distribution lies
// within sigma of its mean (Cantelli), so the median is searched in
// [mu - s - 1, mu + s + 1]; and since E|X - m| <= E|X - mu| <= sigma, Markov's
// inequality leaves at most half of the values at |X - m| >= 2 sigma, so the
// lower median of |X - m| (the MAD) is below 2 sigma and is searched in
// [0, 2 s + 1].  For noise-like rows both windows are under 2048 wide: one
// pass each, three passes in all (five over the full ranges).  The first
// histogram pass of each search also counts the values below its window and
// in it; the selection goes on only if the wanted rank falls inside, which
// makes the result exact whatever the floating-point bound -- otherwise (never
// expected) the same selection runs on the full range.
constexpr int kRT = 512;
constexpr int kRB = 2048;

template <int MODE>  // 0: u = v - base;  1: u = |v - base|   (mod 2^32, no signed overflow)
__device__ __forceinline__ uint32_t robust_key(int32_t v, int32_t base)
{
    if (MODE == 0) return (uint32_t)v - (uint32_t)base;
    return v >= base ? (uint32_t)v - (uint32_t)base : (uint32_t)base - (uint32_t)v;
}

// Calls f(v) for every value of part `part` of `parts` of the row y[0 .. n), spread
// over the block: kRU4 16-byte loads per thread in flight per step; the first
// part also takes the values before the first 16-byte boundary and after the last.
constexpr int kRU4 = 4;
template <typename F>
__device__ __forceinline__ void for_row(const int32_t* __restrict__ y, int64_t n, int part, int parts, F&& f)
{
    const int tid = threadIdx.x;
    int64_t head = (int64_t)(((16u - ((uint32_t)reinterpret_cast<uintptr_t>(y) & 15u)) & 15u) >> 2);
    if (head > n) head = n;
    if (part == 0 && tid < head) f(__ldg(y + tid));
    const int4* y4 = reinterpret_cast<const int4*>(y + head);
    const int64_t n4 = (n - head) >> 2, q1 = n4 * (part + 1) / parts;
    for (int64_t i = n4 * part / parts + tid; i < q1; i += (int64_t)kRT * kRU4) {
        int4 v[kRU4];
#pragma unroll
        for (int u = 0; u < kRU4; u++)
            if (i + u * kRT < q1) v[u] = __ldg(y4 + i + u * kRT);
#pragma unroll
        for (int u = 0; u < kRU4; u++)
            if (i + u * kRT < q1) {
                f(v[u].x);
                f(v[u].y);
                f(v[u].z);
                f(v[u].w);
            }
    }
    const int64_t t0 = head + 4 * n4;
    if (part == 0 && t0 + tid < n) f(__ldg(y + t0 + tid));  // at most 3 values
}

// Block sum of one int64 per thread, returned to every thread (sred: kRT/32 slots).
__device__ __forceinline__ long long block_sum(long long x, long long* sred)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    __syncthreads();  // earlier readers of sred are done
    if (lane == 0) sred[warp] = x;
    __syncthreads();
    long long t = 0;
    for (int i = 0; i < kRT / 32; i++) t += sred[i];
    return t;
}

// Scratch of the selection over a row, by one block or by the blocks of a cluster
// (each one part of the row; every block adds up all blocks' counts through
// distributed shared memory and so takes the same decisions).
struct RobustScratch {
    alignas(16) uint32_t hist[kRB];  // 4 bins a thread (16 bytes)
    uint32_t wsum[kRT / 32];
    int64_t found[2];                // a search's bin (-1: none) and the count before it
    long long sred[kRT / 32];
    int32_t smin[kRT / 32], smax[kRT / 32];
    float ssq[kRT / 32];
    // read by a cluster's other blocks
    long long below, su;             // values below the window; sum of v - y[0]
    int32_t lo, hi;
    double m2;
};
static_assert(kRB == 4 * kRT, "four bins a thread");

// The rank-th smallest key (0-based) among the row's keys in [0, width).  For
// MODE 0, rank counts from the row's smallest value: the first pass counts
// the values under `base` (none when base is the row minimum).  Returns false,
// with every thread agreeing, when the first pass shows the rank outside the
// window.
template <int MODE, bool CLUSTER>
__device__ bool robust_select(const int32_t* __restrict__ y, int64_t n, int part, int parts, int32_t base,
                              uint64_t width, int64_t rank, RobustScratch& sc, uint32_t* out)
{
    uint32_t start = 0;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    bool first = true;
    while (first || width > 1) {
        const int bits = width > 1 ? 64 - __clzll((long long)(width - 1)) : 0;
        const int s = bits > 11 ? bits - 11 : 0;
        reinterpret_cast<uint4*>(sc.hist)[tid] = make_uint4(0u, 0u, 0u, 0u);
        if (tid == 0) sc.found[0] = -1;
        __syncthreads();
        long long below = 0;
        const bool count_below = MODE == 0 && first;
        for_row(y, n, part, parts, [&](int32_t v) {
            const uint32_t k = robust_key<MODE>(v, base);
            if (k >= start && (uint64_t)(k - start) < width) atomicAdd(&sc.hist[(k - start) >> s], 1u);
            else if (count_below && v < base) below++;
        });
        if (count_below) below = block_sum(below, sc.sred);  // syncs the block
        else if (!CLUSTER) __syncthreads();
        uint4 h;
        if (CLUSTER) {
            cg::cluster_group cluster = cg::this_cluster();
            if (tid == 0) sc.below = below;
            cluster.sync();  // every block's counts are complete
            h = make_uint4(0u, 0u, 0u, 0u);
            below = 0;
            for (int r = 0; r < parts; r++) {
                const RobustScratch* o = cluster.map_shared_rank(&sc, r);
                const uint4 c = reinterpret_cast<const uint4*>(o->hist)[tid];
                h.x += c.x;
                h.y += c.y;
                h.z += c.z;
                h.w += c.w;
                if (count_below) below += o->below;
            }
        } else {
            h = reinterpret_cast<const uint4*>(sc.hist)[tid];
        }
        if (count_below) rank -= below;
        // the bin where the running count passes rank (bins in the threads' order)
        const uint32_t own = h.x + h.y + h.z + h.w;
        uint32_t incl = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) sc.wsum[warp] = incl;
        __syncthreads();
        int64_t cum = (int64_t)(incl - own);
        for (int k = 0; k < warp; k++) cum += sc.wsum[k];
        if (cum <= rank && rank < cum + (int64_t)own) {
            int b = 0;
            if (rank >= cum + h.x) cum += h.x, b = 1;
            if (b == 1 && rank >= cum + h.y) cum += h.y, b = 2;
            if (b == 2 && rank >= cum + h.z) cum += h.z, b = 3;
            sc.found[0] = 4 * tid + b;
            sc.found[1] = cum;
        }
        // the answer, and no block clears counts that another still reads
        if (CLUSTER) cg::this_cluster().sync();
        else __syncthreads();
        if (sc.found[0] < 0) return false;  // only on a first pass: later windows hold the rank by construction
        const uint32_t b = (uint32_t)sc.found[0];
        rank -= sc.found[1];
        start += b << s;
        const uint64_t left = width - ((uint64_t)b << s);
        width = left < ((uint64_t)1 << s) ? left : ((uint64_t)1 << s);
        first = false;
        __syncthreads();
    }
    *out = start;
    return true;
}

// Median and MAD of a row in up to three passes (the windows above).
template <bool CLUSTER>
__device__ __noinline__ void row_robust_general(const int32_t* __restrict__ y, int64_t nout, int part_, int parts_,
                                                RobustScratch& sc, af_robust_t* __restrict__ out)
{
    const int part = CLUSTER ? part_ : 0, parts = CLUSTER ? parts_ : 1;
    long long* sred = sc.sred;
    int32_t *smin = sc.smin, *smax = sc.smax;
    float* ssq = sc.ssq;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // pass 1: range, and sums of u = v - y[0] (exact) and of u^2 (fp32 per thread; only the window depends on it)
    const int32_t y0 = __ldg(y);
    int32_t lo = INT32_MAX, hi = INT32_MIN;
    long long su = 0;
    float sq = 0.0f;
    for_row(y, nout, part, parts, [&](int32_t v) {
        lo = min(lo, v);
        hi = max(hi, v);
        su += (long long)v - y0;
        // v - y0 mod 2^32 as a signed value: exact unless the row spans more
        // than 2^31, where only the window estimate (never the result) suffers
        const float f = (float)(int32_t)((uint32_t)v - (uint32_t)y0);
        sq = fmaf(f, f, sq);
    });
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        sq += __shfl_xor_sync(0xffffffffu, sq, o);
    }
    if (lane == 0) {
        smin[warp] = lo;
        smax[warp] = hi;
        ssq[warp] = sq;
    }
    su = block_sum(su, sred);  // syncs: smin, smax, ssq are visible
    lo = smin[0];
    hi = smax[0];
    double m2 = 0.0;
    for (int i = 0; i < kRT / 32; i++) {
        lo = min(lo, smin[i]);
        hi = max(hi, smax[i]);
        m2 += (double)ssq[i];
    }
    if (CLUSTER) {
        cg::cluster_group cluster = cg::this_cluster();
        if (tid == 0) {
            sc.lo = lo;
            sc.hi = hi;
            sc.su = su;
            sc.m2 = m2;
        }
        cluster.sync();
        su = 0;
        m2 = 0.0;
        for (int r = 0; r < parts; r++) {
            const RobustScratch* o = cluster.map_shared_rank(&sc, r);
            lo = min(lo, o->lo);
            hi = max(hi, o->hi);
            su += o->su;
            m2 += o->m2;
        }
    }
    const double nn = (double)nout, mean_u = (double)su / nn;
    m2 /= nn;
    // s >= sigma: the fp32 sums of u^2 (about nout / 512 terms per thread, then 32
    // per warp) carry a relative error below (terms) * 2^-24; the margin is 4x that
    const double rel = 1e-4 + ((double)nout / kRT + 64.0) * 2.4e-7;
    const double sb = sqrt(fmax(m2 - mean_u * mean_u, 0.0) + rel * m2 + 1.0);
    const double mu = (double)y0 + mean_u;
    const int64_t k = (nout - 1) / 2;

    const int64_t wl = max((int64_t)lo, (int64_t)floor(mu - sb) - 1);
    const int64_t wh = min((int64_t)hi, (int64_t)ceil(mu + sb) + 1);
    uint32_t key = 0;
    int32_t med;
    if (wl <= wh && robust_select<0, CLUSTER>(y, nout, part, parts, (int32_t)wl, (uint64_t)(wh - wl) + 1, k, sc, &key))
        med = (int32_t)((uint32_t)(int32_t)wl + key);  // a row value: no overflow in the sum
    else {  // the same selection over the whole range [lo, hi]
        robust_select<0, CLUSTER>(y, nout, part, parts, lo, (uint64_t)((int64_t)hi - lo) + 1, k, sc, &key);
        med = (int32_t)((uint32_t)lo + key);
    }
    const int64_t r2 = max((int64_t)hi - med, (int64_t)med - lo);
    const int64_t wm = min(r2, (int64_t)ceil(2.0 * sb) + 1);
    uint32_t mad = 0;
    if (!robust_select<1, CLUSTER>(y, nout, part, parts, med, (uint64_t)wm + 1, k, sc, &mad))
        robust_select<1, CLUSTER>(y, nout, part, parts, med, (uint64_t)r2 + 1, k, sc, &mad);
    if (tid == 0 && part == 0) {
        out->median = med;
        out->mad = mad;
    }
}

__global__ void __launch_bounds__(kRT, 2) k_row_robust(const int32_t* __restrict__ Y, int64_t nout,
                                                    af_robust_t* __restrict__ out)
{
    __shared__ RobustScratch sc;
    row_robust_general<false>(Y + (int64_t)blockIdx.x * nout, nout, 0, 1, sc, out + blockIdx.x);
}

// ---- long rows: one pass.  A sample of 4096 values (1024 16-byte pieces, one at a
// scattered place in each of as many equal stretches) gives estimates m of the
// median and M of the MAD, good to a few hundredths of sigma on any smooth
// distribution.  One pass over the row then
// counts, at unit resolution, the values in three windows -- around m, m - M
// and m + M, each a few estimate errors wide -- and the values below each
// window.  Cumulative counts C(z) = #(v < z) are therefore exact for z inside a
// window, and the exact median (the value holding rank k = (n - 1) / 2) and MAD
// (the smallest x with C(med + x + 1) - C(med - x) > k) follow without another
// pass: both are checked against the windows' edges, and a row whose answer
// lies outside them (none seen on noise) takes the general selection.  Where
// the windows meet (M of a few units) one dense window covers them all.  A row
// whose windows would not fit the bins (M above some 11,000; noise that fills the
// bytes of 40,000 channels stays below), or whose sample has too few values near its
// median to trust that estimate (two far-apart modes), goes to the general selection
// without that pass.
// A cluster of blocks shares a row, each counting one part; the first block
// adds up the others' counts through distributed shared memory.  The general
// selection is shared as well where the sample asks for it (left to the first block,
// 500 x 200001 rows that need it took 880 us, 540 so; called there and not after the
// pass, whose rows it would slow down by 2 to 6 %).  Bound by issue
// (about 25 instructions per 32 values, the three window tests and counts) and
// HBM: 1001 x 215261 plane 0.53 ms in three passes, 0.24 ms in one.
// Rows below 16384 values keep the general selection: the sample would be a
// quarter of the row and more.
constexpr int kRS = 4096;                 // sample values
constexpr int64_t kRobustOnePass = 16384; // shortest row for the one-pass kernel
constexpr int kRH = 12288;                // histogram bins of all windows (48 KB: M up to 11,000)

struct RobustOnePass {
    union {
        RobustScratch gen;
        struct {
            alignas(16) uint32_t hist[kRH];  // counts per bin, then exclusive prefix sums (read 16 bytes at a time)
            uint32_t wsum[kRT / 32];
            uint32_t below[3];            // values below each window (of this block's part)
            uint32_t near[kRT / 32];      // per warp: sample values near the median, two counts a word
            int32_t lo, hi;               // sample range
            uint32_t bin, cum;            // a search's answer
            int32_t med, mad;
            int ok;
        } one;
    };
};

// Block-wide: the bin of hist[0 .. 4 kRT) where the running count passes rank
// and the count before it, in sc.bin and sc.cum.
__device__ __forceinline__ void find_rank(RobustOnePass& sc, uint32_t rank)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint4 h = *reinterpret_cast<const uint4*>(sc.one.hist + 4 * tid);
    const uint32_t own = h.x + h.y + h.z + h.w;
    uint32_t incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) sc.one.wsum[warp] = incl;
    __syncthreads();
    uint32_t cum = incl - own;
    for (int k = 0; k < warp; k++) cum += sc.one.wsum[k];
    if (cum <= rank && rank < cum + own) {
        const uint32_t hv[4] = {h.x, h.y, h.z, h.w};
        int j = 0;
        while (rank >= cum + hv[j]) cum += hv[j++];
        sc.one.bin = 4 * tid + j;
        sc.one.cum = cum;
    }
    __syncthreads();
}

// Estimate (lower median of the sample's keys, to within *res) by at most two
// histogram passes of 2048 bins over [0, range].
__device__ __forceinline__ uint32_t sample_median(const uint32_t (&key)[kRS / kRT], uint32_t range, RobustOnePass& sc,
                                                  uint32_t* res)
{
    const int tid = threadIdx.x;
    uint32_t start = 0, rank = (kRS - 1) / 2;
    int s = max(0, 21 - __clz(range));  // bins of 2^s: range >> s < 2048
    for (int pass = 0; pass < 2; pass++) {
        *reinterpret_cast<uint4*>(sc.one.hist + 4 * tid) = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kRS / kRT; j++) {
            const uint32_t b = (key[j] - start) >> s;
            if (key[j] >= start && b < (uint32_t)kRB) atomicAdd(&sc.one.hist[b], 1u);
        }
        __syncthreads();
        find_rank(sc, rank);
        start += sc.one.bin << s;
        rank -= sc.one.cum;
        __syncthreads();
        if (s == 0) break;
        if (pass == 0) s = max(0, s - 11);
    }
    *res = s == 0 ? 0u : (1u << s);
    return start;
}

// The general selection of a cluster's row by all of its blocks.
__device__ __noinline__ void row_robust_shared(const int32_t* __restrict__ Y, int64_t nout, af_robust_t* __restrict__ out)
{
    extern __shared__ __align__(16) uint8_t robust_smem[];
    cg::cluster_group cluster = cg::this_cluster();
    const int parts = (int)cluster.num_blocks(), part = (int)cluster.block_rank();
    const int64_t d = blockIdx.x / parts;
    row_robust_general<true>(Y + d * nout, nout, part, parts, reinterpret_cast<RobustOnePass*>(robust_smem)->gen, out + d);
}

__global__ void __launch_bounds__(kRT, 2)
k_row_robust1(const int32_t* __restrict__ Y, int64_t nout, af_robust_t* __restrict__ out)
{
    extern __shared__ __align__(16) uint8_t robust_smem[];
    RobustOnePass& sc = *reinterpret_cast<RobustOnePass*>(robust_smem);
    cg::cluster_group cluster = cg::this_cluster();
    const int parts = (int)cluster.num_blocks(), part = (int)cluster.block_rank();
    const int64_t d = blockIdx.x / parts;
    const int32_t* y = Y + d * nout;
    const int tid = threadIdx.x, lane = tid & 31;
    const int64_t head = (int64_t)(((16u - ((uint32_t)reinterpret_cast<uintptr_t>(y) & 15u)) & 15u) >> 2);
    const int4* y4 = reinterpret_cast<const int4*>(y + head);
    const int64_t n4 = (nout - head) >> 2;

    // the sample, its range
    int32_t sv[kRS / kRT];
    {
        const int64_t step = n4 / (kRS / 4);
#pragma unroll
        for (int j = 0; j < kRS / kRT / 4; j++) {
            const uint32_t piece = tid + j * kRT;  // even steps would see one phase of a periodic row
            const int4 v = __ldg(y4 + piece * step + __umulhi(piece * 2654435761u, (uint32_t)step));
            sv[4 * j] = v.x;
            sv[4 * j + 1] = v.y;
            sv[4 * j + 2] = v.z;
            sv[4 * j + 3] = v.w;
        }
    }
    if (tid == 0) {
        sc.one.lo = INT32_MAX;
        sc.one.hi = INT32_MIN;
        sc.one.below[0] = sc.one.below[1] = sc.one.below[2] = 0u;
    }
    __syncthreads();
    int32_t lo = sv[0], hi = sv[0];
#pragma unroll
    for (int j = 1; j < kRS / kRT; j++) {
        lo = min(lo, sv[j]);
        hi = max(hi, sv[j]);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) {
        atomicMin(&sc.one.lo, lo);
        atomicMax(&sc.one.hi, hi);
    }
    __syncthreads();
    lo = sc.one.lo;
    hi = sc.one.hi;
    uint32_t key[kRS / kRT], res, rmad;
#pragma unroll
    for (int j = 0; j < kRS / kRT; j++) key[j] = (uint32_t)sv[j] - (uint32_t)lo;
    const uint32_t mk = sample_median(key, (uint32_t)hi - (uint32_t)lo, sc, &res);
    const int32_t m = (int32_t)((uint32_t)lo + mk);
#pragma unroll
    for (int j = 0; j < kRS / kRT; j++) key[j] = sv[j] >= m ? (uint32_t)sv[j] - (uint32_t)m : (uint32_t)m - (uint32_t)sv[j];
    const uint32_t M = sample_median(key, max((uint32_t)hi - (uint32_t)m, (uint32_t)m - (uint32_t)lo), sc, &rmad);

    // windows: 5 standard errors of a normal sample's estimates (0.029 M and 0.034 M) and the estimates' resolution
    const bool sane = M < (1u << 20) && res < (1u << 20) && rmad < (1u << 20);
    const int32_t dc = (int32_t)(M / 7) + 2 + (int32_t)min(res, 1u << 20);
    const int32_t dw = (int32_t)(M / 5) + 2 + (int32_t)min(res + rmad, 1u << 20);
    const int32_t in = (int32_t)min(M, 1u << 20) - dw, outer = (int32_t)min(M, 1u << 20) + dw;  // |v - m| of the outer windows
    const bool dense = in <= dc;
    const int64_t bins = dense ? 2 * (int64_t)outer + 1 : 2 * (int64_t)dc + 1 + 2 * (2 * (int64_t)dw + 1);
    // windows inside the int32 range, so that (v - start) mod 2^32 < width exactly for the values in them
    const bool inside = sane && bins <= kRH && (int64_t)m - outer >= INT32_MIN && (int64_t)m + outer < INT32_MAX;
    // The median's rank must fall into its window: some values between the estimate and the window's edges, in a quarter
    // of the sample from all over the row (a normal one has 39 +- 6 on either side, and the rank an error of 8 there).
    bool fits = inside;
    if (inside) {  // the same in every thread
        const uint32_t wm = dense ? outer : dc;
        auto near = [&](int j) -> uint32_t {  // at or below m | at or above
            return key[j] > wm ? 0u : (sv[j] <= m ? 1u : 0u) + (sv[j] >= m ? 1u << 16 : 0u);
        };
        const uint32_t c = __reduce_add_sync(0xffffffffu, near(0) + near(kRS / kRT / 2));
        if (lane == 0) sc.one.near[tid >> 5] = c;
        __syncthreads();
        const uint32_t n = __reduce_add_sync(0xffffffffu, sc.one.near[lane & 15]) >> 1;  // every warp's count twice
        fits = min(n & 0xFFFFu, n >> 16) >= 16;
    }
    if (!fits && parts > 1) {  // the same in every block of the cluster
        __syncthreads();       // the scratch is the general selection's now
        row_robust_shared(Y, nout, out);
        return;
    }
    // window starts (as v - m), widths and first bins: below m - M, around m, above m + M; dense: the first alone
    const int32_t w0 = -outer, w1 = -dc, w2 = in;
    const int nb0 = dense ? 2 * outer + 1 : 2 * dw + 1, nb1 = dense ? 0 : 2 * dc + 1, nb2 = dense ? 0 : 2 * dw + 1;
    if (fits) {
        for (int i = tid; i < nb0 + nb1 + nb2; i += kRT) sc.one.hist[i] = 0u;
        __syncthreads();
        uint32_t b0 = 0, b1 = 0, b2 = 0;
        // shared address of value v's bin: 4 v + k0, k1 or k2 (mod 2^32) by its window
        const uint32_t s0 = (uint32_t)(m + w0), s1 = (uint32_t)(m + w1), s2 = (uint32_t)(m + w2);
        const uint32_t hb = (uint32_t)__cvta_generic_to_shared(sc.one.hist);
        const uint32_t k0 = hb - 4u * s0, k1 = hb + 4u * ((uint32_t)nb0 - s1), k2 = hb + 4u * ((uint32_t)(nb0 + nb1) - s2);
        auto count = [&](int32_t v) {  // dense: windows 1 and 2 are empty, their counts are not used
            asm volatile(
                "{\n\t.reg .pred p, q, r;\n\t.reg .u32 a, k;\n\t"
                "setp.lt.s32 p, %3, %4;\n\t@p add.u32 %0, %0, 1;\n\t"
                "setp.lt.s32 p, %3, %5;\n\t@p add.u32 %1, %1, 1;\n\t"
                "setp.lt.s32 p, %3, %6;\n\t@p add.u32 %2, %2, 1;\n\t"
                "sub.u32 a, %3, %4;\n\tsetp.lt.u32 p, a, %7;\n\t"
                "sub.u32 a, %3, %5;\n\tsetp.lt.or.u32 q, a, %8, p;\n\t"
                "sub.u32 a, %3, %6;\n\tsetp.lt.or.u32 r, a, %9, q;\n\t"
                "selp.u32 k, %11, %12, q;\n\tselp.u32 k, %10, k, p;\n\t"
                "mad.lo.u32 a, %3, 4, k;\n\t@r red.shared.add.u32 [a], 1;\n\t}"
                : "+r"(b0), "+r"(b1), "+r"(b2)
                : "r"(v), "r"(s0), "r"(s1), "r"(s2), "r"(nb0), "r"(nb1), "r"(nb2), "r"(k0), "r"(k1), "r"(k2)
                : "memory");
        };
        // this block's part of the row, in 16-byte pieces; the first block also takes the row's unaligned ends
        const int64_t q0 = n4 * part / parts, q1 = n4 * (part + 1) / parts;
        const int4* p = y4 + q0 + tid;
        const int steps = (int)((q1 - q0) / (kRT * kRU4));  // whole steps of the block
        for (int f = 0; f < steps; f++, p += kRT * kRU4) {
            int4 v[kRU4];
#pragma unroll
            for (int u = 0; u < kRU4; u++) v[u] = __ldg(p + u * kRT);
#pragma unroll
            for (int u = 0; u < kRU4; u++) {
                count(v[u].x);
                count(v[u].y);
                count(v[u].z);
                count(v[u].w);
            }
        }
        for (const int4* e = y4 + q1; p < e; p += kRT) {  // at most kRU4 - 1 pieces a thread
            const int4 t = __ldg(p);
            count(t.x);
            count(t.y);
            count(t.z);
            count(t.w);
        }
        if (part == 0) {
            if (tid < head) count(__ldg(y + tid));
            const int64_t t0 = head + 4 * n4;
            if (t0 + tid < nout) count(__ldg(y + t0 + tid));  // at most 3 values
        }
        b0 = __reduce_add_sync(0xffffffffu, b0);
        b1 = __reduce_add_sync(0xffffffffu, b1);
        b2 = __reduce_add_sync(0xffffffffu, b2);
        if (lane == 0) {
            atomicAdd(&sc.one.below[0], b0);
            atomicAdd(&sc.one.below[1], b1);
            atomicAdd(&sc.one.below[2], b2);
        }
    }
    cluster.sync();  // every block's counts are final (all blocks of a cluster share the windows: same sample)
    bool done = false;
    if (part == 0 && fits) {
        const int nb = nb0 + nb1 + nb2;
        for (int q = 1; q < parts; q++) {
            const RobustOnePass* r = cluster.map_shared_rank(&sc, q);
            for (int i = tid; i < nb; i += kRT) sc.one.hist[i] += r->one.hist[i];
            if (tid < 3) sc.one.below[tid] += r->one.below[tid];
        }
        if (tid == 0) sc.one.ok = 0;
        __syncthreads();
        // exclusive prefix sums of the bins, in place, 4 kRT at a time
        const int warp = tid >> 5;
        uint32_t base = 0;
        for (int c0 = 0; c0 < nb; c0 += 4 * kRT) {
            const int i = c0 + 4 * tid;
            uint32_t h[4];
#pragma unroll
            for (int j = 0; j < 4; j++) h[j] = i + j < nb ? sc.one.hist[i + j] : 0u;
            const uint32_t own = h[0] + h[1] + h[2] + h[3];
            uint32_t incl = own;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            if (lane == 31) sc.one.wsum[warp] = incl;
            __syncthreads();
            uint32_t e = base + incl - own;
            for (int k = 0; k < warp; k++) e += sc.one.wsum[k];
            for (int k = 0; k < kRT / 32; k++) base += sc.one.wsum[k];
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (i + j < nb) {
                    sc.one.hist[i + j] = e;
                    e += h[j];
                }
            __syncthreads();  // wsum is read before the next chunk writes it
        }
        // C(z) - (values below window s) for z = window start + i, 0 <= i <= its bins
        const uint32_t total = base;
        auto cnt = [&](int s, int i) -> int64_t {
            const int first = s == 0 ? 0 : s == 1 ? nb0 : nb0 + nb1;
            const uint32_t e = first + i < nb ? sc.one.hist[first + i] : total;
            return (int64_t)sc.one.below[s] + (int64_t)(e - sc.one.hist[first]);
        };
        const int64_t k = (nout - 1) / 2;
        const int sm = dense ? 0 : 1, nbm = dense ? nb0 : nb1, wm = dense ? w0 : w1;
        // the median: the bin of its window that holds rank k
        for (int i = tid; i < nbm; i += kRT)
            if (cnt(sm, i) <= k && k < cnt(sm, i + 1)) {
                sc.one.med = wm + i;
                sc.one.ok = 1;
            }
        __syncthreads();
        if (sc.one.ok == 1) {
            const int med = sc.one.med;  // relative to m
            // N(x) = C(med + x + 1) - C(med - x) = #(|v - median| <= x), for x with both ends inside their windows
            const int sl = 0, sr = dense ? 0 : 2, wr = dense ? w0 : w2, nbr = dense ? nb0 : nb2;
            const int xlo = dense ? -1 : max(wr - med - 1, med - (w0 + nb0));
            const int xhi = min(wr + nbr - med - 1, med - w0);
            auto N = [&](int x) -> int64_t { return x < 0 ? 0 : cnt(sr, med + x + 1 - wr) - cnt(sl, med - x - w0); };
            for (int x = xlo + 1 + tid; x <= xhi; x += kRT)
                if (N(x) > k && N(x - 1) <= k) {
                    sc.one.mad = x;
                    sc.one.ok = 2;
                }
        }
        __syncthreads();
        if (sc.one.ok == 2) {
            done = true;
            if (tid == 0) {
                out[d].median = (int32_t)((uint32_t)m + (uint32_t)sc.one.med);
                out[d].mad = sc.one.mad;
            }
        }
        __syncthreads();
    }
    cluster.sync();  // the first block has read the others' shared memory
    if (part == 0 && !done) row_robust_general<false>(y, nout, 0, 1, sc.gen, out + d);
}

// Robust S/N constants: snr = (B - w*med) * k, k = 1/(1.482602218505602 * mad * sqrt(w)).
__global__ void k_rowconst_robust(const af_robust_t* __restrict__ r, int ndm, af_widths_t w,
                                  af_rowconst_t* __restrict__ rc)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ndm * w.n) return;
    const int d = i / w.n, wi = i % w.n;
    const int64_t W = w.w[wi];
    const double sigma = 1.482602218505602 * (double)r[d].mad;
    af_rowconst_t o;
    o.q = W * r[d].median;
    o.k = sigma > 0.0 ? (float)(1.0 / (sigma * sqrt((double)W))) : 0.0f;
    o.c = 0.0f;
    rc[(int64_t)d * AF_MAX_WIDTHS + wi] = o;
}

}  // namespace

int af_launch_row_robust(const int32_t* d_plane, int ndm, int64_t nout, af_robust_t* d_robust, cudaStream_t s)
{
    if (nout < kRobustOnePass || nout > INT32_MAX) {
        k_row_robust<<<ndm, kRT, 0, s>>>(d_plane, nout, d_robust);
        return af_cuda_check(cudaGetLastError(), "robust row statistics launch");
    }
    // blocks per row: enough for four waves of two per SM, each with at least 16384 values
    int dev = 0, nsm = 0;
    AF_CUDA(cudaGetDevice(&dev));
    AF_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    int parts = 1;
    while (parts < 8 && (int64_t)ndm * parts < 8 * nsm && nout / (2 * parts) >= 16384) parts *= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(ndm * parts));
    cfg.blockDim = dim3(kRT);
    cfg.dynamicSmemBytes = sizeof(RobustOnePass);
    cfg.stream = s;
    if (int rc = af_ensure_smem((const void*)k_row_robust1, sizeof(RobustOnePass))) return rc;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)parts;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return af_cuda_check(cudaLaunchKernelEx(&cfg, k_row_robust1, d_plane, nout, d_robust),
                         "robust row statistics launch");
}

int af_launch_boxcar_robust(const int32_t* d_plane, int ndm, int64_t nout, const af_robust_t* d_robust,
                            const af_widths_t& w, af_rowconst_t* d_rowconst, float* d_best_snr, uint8_t* d_best_w,
                            cudaStream_t s)
{
    const int nrc = ndm * w.n;
    k_rowconst_robust<<<(nrc + 255) / 256, 256, 0, s>>>(d_robust, ndm, w, d_rowconst);
    if (int rc = af_cuda_check(cudaGetLastError(), "robust rowconst launch")) return rc;
    return launch_boxcar_tiles(d_plane, ndm, nout, w, d_rowconst, d_best_snr, d_best_w, s);
}

int af_launch_boxcar(const int32_t* d_plane, int ndm, int64_t nout, const af_rowstats_t* d_stats,
                     const af_widths_t& w, af_rowconst_t* d_rowconst, float* d_best_snr, uint8_t* d_best_w,
                     cudaStream_t s)
{
    const int nrc = ndm * w.n;
    k_rowconst<<<(nrc + 255) / 256, 256, 0, s>>>(d_stats, ndm, nout, w, d_rowconst);
    if (int rc = af_cuda_check(cudaGetLastError(), "rowconst launch")) return rc;
    return launch_boxcar_tiles(d_plane, ndm, nout, w, d_rowconst, d_best_snr, d_best_w, s);
}
