// grid.cu -- DM-time slice gridding for an image detector (Sec. 2.4,
// "Griding and Rendering"): the plane's time axis is cut into slices of ns
// columns, each slice resampled to an M x M image and normalised to 8 bits.
//
//   area path (ndm > M and slice width w > M): exact pixel-area mean,
//     W(i,j) = sum_r sum_c ovr(i,r) ovc(j,c) X[r][c0 + c]   (int64, exact),
//     ovr(i,r) = |[i ndm, (i+1) ndm) & [r M, (r+1) M)|, ovc likewise with w;
//     U = W / (ndm w).
//   Lanczos-4 path otherwise: separable, source x = (i + 0.5) n / M - 0.5, taps
//     floor(x) - 3 .. floor(x) + 4, L(t) = sinc(t) sinc(t/4) normalised,
//     replicated border; evaluated in double.
//   Y = floor(255 (U - umin) / (umax - umin + eps) + 1/2), eps = 1e-6, on the
//     Lanczos path; on the area path exactly from the integers W, without eps
//     (0 for a constant slice).
//
// Two passes over the plane: the first finds each slice's min and max
// (block reduction + 64-bit atomics into the caller's work array), the
// second recomputes the values and writes Y, its blocks in reverse order so
// that it begins with what the first left in L2.
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "internal.h"

namespace {

constexpr int kGT = 256;

// Monotone int64 key of a double (for atomic min / max).
__device__ __forceinline__ long long dkey(double v)
{
    const long long b = __double_as_longlong(v);
    return b >= 0 ? b : b ^ 0x7FFFFFFFFFFFFFFFLL;
}
__device__ __forceinline__ double dval(long long k)
{
    return __longlong_as_double(k >= 0 ? k : k ^ 0x7FFFFFFFFFFFFFFFLL);
}

// Block-wide minimum and maximum into the slice's pair of the work array.
__device__ __forceinline__ void slice_minmax(long long lo, long long hi, long long* work)
{
    __shared__ long long slo[kGT / 32], shi[kGT / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if ((threadIdx.x & 31) == 0) {
        slo[threadIdx.x >> 5] = lo;
        shi[threadIdx.x >> 5] = hi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < kGT / 32; k++) {
            lo = min(lo, slo[k]);
            hi = max(hi, shi[k]);
        }
        atomicMin(work, lo);
        atomicMax(work + 1, hi);
    }
}

// floor((510 a + r) / (2 r)), 0 <= a <= r, r > 0: from a float estimate (within
// one) and exact 64-bit tests where 512 r fits, else by 128-bit division.
__device__ __forceinline__ uint32_t gray(unsigned long long a, unsigned long long r)
{
    if (r >> 54) return (uint32_t)((510 * (unsigned __int128)a + r) / (2 * (unsigned __int128)r));
    const unsigned long long num = 510 * a + r, den = 2 * r;
    uint32_t y = (uint32_t)(255.0f * __fdividef((float)a, (float)r) + 0.5f);
    if (y * den > num) y--;
    else if ((y + 1) * den <= num) y++;
    return y;
}

// Area path by columns, for wide pixels.  Block = (slice, output row i, run of kGT
// output columns): the plane rows that row i covers are added, weighted, column by
// column with coalesced loads into V[c] = sum_r ovr(i, r) X[r][c] (shared memory, as
// many columns at a time as fit), and thread j sums its pixel's columns from there,
// the first and last weighted.  V is int32: valid while every value of the block's
// columns is non-negative and (their bitwise or) x h is below 2^31 (planes of 8-bit
// sums); otherwise the block starts again with int64, in pass 1 at once where the
// slice's sums show that int32 would not do.
// PASS 0: min / max into work; PASS 1: write Y.
// Bound by HBM (the plane twice).  22 slices of 1001 x 10173 to 512 x 512: a pass
// took 0.42 ms with every pixel loading its own 20 columns of 2 to 3 rows (lanes
// 80 bytes apart) and 64-bit divisions per pixel, 0.23 ms so
// (latency: a block's loads, sums and reduction follow one another; rows staged by
// asynchronous copies in 128-thread blocks took the same).
constexpr int kGU = 5;                    // columns per thread and step
constexpr int kGCBytes = 5632 * 4;        // shared memory for V, at most

struct AreaRows {
    const int32_t* x;      // row r_lo, first column of the slice
    int64_t nout;
    int n, lo, hi, M;      // rows, weights of the first and last, of the others
};

// One step of kGU columns c, c + kGT, ...: adds rows at p0, p1, p2 (first column
// c of each) with their weights, all loads first.  CHECK: columns from n on do
// not exist.
template <typename T, bool CHECK>
__device__ __forceinline__ int32_t area_step(const int32_t* p0, const int32_t* p1, const int32_t* p2, int o0, int o1,
                                             int o2, int c, int n, T (&v)[kGU])
{
    int32_t y[3][kGU], any = 0;
#pragma unroll
    for (int u = 0; u < kGU; u++) {
        const bool in = !CHECK || c + u * kGT < n;
        y[0][u] = in ? __ldg(p0 + u * kGT) : 0;
        y[1][u] = in ? __ldg(p1 + u * kGT) : 0;
        y[2][u] = in ? __ldg(p2 + u * kGT) : 0;
    }
#pragma unroll
    for (int u = 0; u < kGU; u++) {
        any |= y[0][u] | y[1][u];
        any |= y[2][u];
        v[u] += (T)o0 * y[0][u] + (T)o1 * y[1][u] + (T)o2 * y[2][u];
    }
    return any;
}

// V[c] of columns c0 .. c0 + n - 1 into shared memory; returns the or of the
// values read.  Rows are taken three at a time (a missing one repeats the last
// row with weight 0); up to three rows (images of up to twice as many DMs as
// rows) need no loop over them.
template <typename T>
__device__ __forceinline__ int32_t area_columns(const AreaRows& a, int c0, int n, T* V)
{
    const int tid = (int)threadIdx.x;
    int32_t any = 0;
    auto weight = [&](int k) { return k == 0 ? a.lo : k < a.n - 1 ? a.M : k == a.n - 1 ? a.hi : 0; };
    const int32_t* x = a.x + c0 + tid;
    if (a.n <= 3) {
        const int32_t *p0 = x, *p1 = x + (int64_t)min(1, a.n - 1) * a.nout, *p2 = x + (int64_t)min(2, a.n - 1) * a.nout;
        const int o0 = weight(0), o1 = weight(1), o2 = weight(2);
        int c = tid;
        for (; c + (kGU - 1) * kGT < n; c += kGU * kGT, p0 += kGU * kGT, p1 += kGU * kGT, p2 += kGU * kGT) {
            T v[kGU] = {};
            any |= area_step<T, false>(p0, p1, p2, o0, o1, o2, c, n, v);
#pragma unroll
            for (int u = 0; u < kGU; u++) V[c + u * kGT] = v[u];
        }
        if (c < n) {
            T v[kGU] = {};
            any |= area_step<T, true>(p0, p1, p2, o0, o1, o2, c, n, v);
#pragma unroll
            for (int u = 0; u < kGU; u++)
                if (c + u * kGT < n) V[c + u * kGT] = v[u];
        }
        return any;
    }
    for (int c = tid; c < n; c += kGU * kGT, x += kGU * kGT) {
        T v[kGU] = {};
        for (int r = 0; r < a.n; r += 3)
            any |= area_step<T, true>(x + (int64_t)r * a.nout, x + (int64_t)min(r + 1, a.n - 1) * a.nout,
                                      x + (int64_t)min(r + 2, a.n - 1) * a.nout, weight(r), weight(r + 1), weight(r + 2),
                                      c, n, v);
#pragma unroll
        for (int u = 0; u < kGU; u++)
            if (c + u * kGT < n) V[c + u * kGT] = v[u];
    }
    return any;
}

// a / M; small: a < 2^32, where a 64-bit division would take several times as long.
__device__ __forceinline__ int div_m(long long a, int M, bool small)
{
    return small ? (int)((uint32_t)a / (uint32_t)M) : (int)(a / M);
}

// W of pixel (i, j) of the slice that starts at column c0: its rows and columns
// with their weights, in 64 bits.
__device__ __forceinline__ long long area_pixel(const int32_t* __restrict__ X, int64_t nout, int h, int64_t c0, int w,
                                                int M, int i, int j, bool small)
{
    const long long ri0 = (long long)i * h, ri1 = ri0 + h, cj0 = (long long)j * w, cj1 = cj0 + w;
    const int r_lo = div_m(ri0, M, small), r_hi = div_m(ri1 - 1, M, small);
    const int c_lo = div_m(cj0, M, small), c_hi = div_m(cj1 - 1, M, small);
    // weights of the first and last row and column, M of the others
    const int rl = (int)(min(ri1, (long long)(r_lo + 1) * M) - ri0), rh = (int)(ri1 - (long long)r_hi * M);
    const int cl = (int)(min(cj1, (long long)(c_lo + 1) * M) - cj0), ch = (int)(cj1 - (long long)c_hi * M);
    const int32_t* x = X + (int64_t)r_lo * nout + c0;
    long long W = 0;
    for (int r = r_lo; r <= r_hi; r++, x += nout) {
        long long row = (long long)cl * __ldg(x + c_lo);
        for (int c = c_lo + 1; c < c_hi; c++) row += (long long)M * __ldg(x + c);
        if (c_hi > c_lo) row += (long long)ch * __ldg(x + c_hi);
        W += row * (r == r_lo ? rl : r == r_hi ? rh : M);
    }
    return W;
}

template <int PASS>
__global__ void __launch_bounds__(kGT, 4)
k_grid_area(const int32_t* __restrict__ X, int h, int64_t nout, int64_t ns, int s0, int M, unsigned runs, int cols,
            long long* __restrict__ work, uint8_t* __restrict__ out)
{
    extern __shared__ long long smem[];  // cols int32
    const unsigned blk = PASS == 0 ? blockIdx.x : gridDim.x - 1 - blockIdx.x;
    const int i = (int)(blk / runs % (unsigned)M), s = s0 + (int)(blk / runs / (unsigned)M);
    const int j0 = (int)(blk % runs) * kGT, j = j0 + (int)threadIdx.x;
    const int64_t c0 = (int64_t)s * ns;
    const int w = (int)min(ns, nout - c0);
    const long long ri0 = (long long)i * h, ri1 = ri0 + h;
    const bool small = (long long)M * max(h, w) + w < (1LL << 32);
    const int r_lo = div_m(ri0, M, small), r_hi = div_m(ri1 - 1, M, small);
    AreaRows rows;
    rows.x = X + c0 + (int64_t)r_lo * nout;
    rows.nout = nout;
    rows.n = r_hi - r_lo + 1;
    rows.lo = (int)(min(ri1, (long long)(r_lo + 1) * M) - ri0);
    rows.hi = (int)(ri1 - (long long)r_hi * M);
    rows.M = M;
    // the pixel's columns [cj0, cj1) / M, the block's
    const long long cj0 = (long long)j * w, cj1 = cj0 + w;
    const bool in = j < M;
    const int c_lo = in ? div_m(cj0, M, small) : 0, c_hi = in ? div_m(cj1 - 1, M, small) : 0;
    const int b_lo = div_m((long long)j0 * w, M, small), b_hi = div_m((long long)min(j0 + kGT, M) * w - 1, M, small);
    // weights of the parts of the pixel's first and last column outside it
    const int out_lo = (int)(cj0 - (long long)c_lo * M), out_hi = (int)((long long)(c_hi + 1) * M - cj1);
    long long W = 0;
    // adds the pixel's part of columns k0 .. k0 + n - 1 (modulo 2^64: the pixel's sum fits, its parts may not)
    auto add = [&](const auto* V, int k0, int n) {
        const int a = max(c_lo, k0), e = min(c_hi, k0 + n - 1);
        unsigned long long sum = 0;
        for (int c = a; c <= e; c++) sum += (unsigned long long)((long long)V[c - k0] * M);
        if (a == c_lo && a <= e) sum -= (unsigned long long)((long long)V[c_lo - k0] * out_lo);
        if (e == c_hi && a <= e) sum -= (unsigned long long)((long long)V[c_hi - k0] * out_hi);
        W = (long long)((unsigned long long)W + sum);
    };
    const long long lo = PASS == 1 ? work[2 * s] : 0, hi = PASS == 1 ? work[2 * s + 1] : 0;
    bool wide = lo < 0 || hi > (long long)w << 31;  // hi / w: the slice's largest mean column sum
    for (int k0 = b_lo; k0 <= b_hi && !wide; k0 += cols) {
        const int n = min(cols, b_hi + 1 - k0);
        int32_t* V = reinterpret_cast<int32_t*>(smem);
        if (k0 > b_lo) __syncthreads();  // the last columns are read
        const int32_t any = area_columns(rows, k0, n, V);
        wide = __syncthreads_or(any < 0 || (long long)any * h > INT32_MAX);
        if (!wide && j < M) add(V, k0, n);
    }
    if (wide) {
        W = 0;
        for (int k0 = b_lo; k0 <= b_hi; k0 += cols / 2) {
            const int n = min(cols / 2, b_hi + 1 - k0);
            __syncthreads();
            area_columns(rows, k0, n, smem);
            __syncthreads();
            if (j < M) add(smem, k0, n);
        }
    }
    if (PASS == 0) {
        slice_minmax(j < M ? W : LLONG_MAX, j < M ? W : LLONG_MIN, work + 2 * s);
    } else if (j < M) {
        const unsigned long long rng = (unsigned long long)(hi - lo);
        out[((int64_t)s * M + i) * M + j] = rng == 0 ? (uint8_t)0 : (uint8_t)gray((unsigned long long)(W - lo), rng);
    }
}

// Area path pixel by pixel, for narrow pixels.  Block = (slice, run of kGT of its
// M x M pixels), thread = pixel: no shared memory, no barriers but the reduction's,
// and no lane idle however small M is.  Bound by the loads' latency and the sums.
// 257 x 257 to 256 x 256, 605 slices: 334 us by columns (343 with 64-bit divisions), 190 so;
// 3 x 7 to 2 x 2, 200,000 slices: 3016 us by columns (1491), 493 so.
template <int PASS>
__global__ void __launch_bounds__(kGT)
k_grid_pixel(const int32_t* __restrict__ X, int h, int64_t nout, int64_t ns, int s0, int M, unsigned runs,
             long long* __restrict__ work, uint8_t* __restrict__ out)
{
    const unsigned blk = PASS == 0 ? blockIdx.x : gridDim.x - 1 - blockIdx.x;
    const int s = s0 + (int)(blk / runs), e = (int)(blk % runs) * kGT + (int)threadIdx.x;
    const int64_t c0 = (int64_t)s * ns;
    const int w = (int)min(ns, nout - c0);
    const bool in = e < M * M, small = (long long)M * max(h, w) + w < (1LL << 32);
    const int i = e / M;
    const long long W = in ? area_pixel(X, nout, h, c0, w, M, i, e - i * M, small) : 0;
    if (PASS == 0) {
        slice_minmax(in ? W : LLONG_MAX, in ? W : LLONG_MIN, work + 2 * s);
    } else if (in) {
        const long long lo = work[2 * s];
        const unsigned long long rng = (unsigned long long)(work[2 * s + 1] - lo);
        out[(int64_t)s * M * M + e] = rng == 0 ? (uint8_t)0 : (uint8_t)gray((unsigned long long)(W - lo), rng);
    }
}

// Lanczos-4 taps of output index i for an axis of n input samples.
__device__ __forceinline__ int lanczos_taps(int i, int n, int M, double* wt)
{
    const double x = ((double)i + 0.5) * (double)n / (double)M - 0.5;
    const int k0 = (int)floor(x);
    double tot = 0.0;
#pragma unroll
    for (int a = 0; a < 8; a++) {
        const double t = x - (double)(k0 - 3 + a);
        double v;
        if (t == 0.0) {
            v = 1.0;
        } else {
            const double pt = 3.141592653589793 * t;
            v = (sinpi(t) / pt) * (sinpi(t * 0.25) / (pt * 0.25));
        }
        wt[a] = v;
        tot += v;
    }
#pragma unroll
    for (int a = 0; a < 8; a++) wt[a] /= tot;
    return k0 - 3;
}

__global__ void k_grid_init(long long* work, int S)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < S) {
        work[2 * s] = LLONG_MAX;
        work[2 * s + 1] = LLONG_MIN;
    }
}

// Lanczos path.  Block = (slice, ti output rows, kLJ output columns).  Both axes'
// taps are computed once per block into shared memory (fp64 sines and
// divisions: on this chip the dearest part), then the horizontal sums H[r][j] of
// the plane rows the block needs, then each pixel's vertical sum over 8 of them;
// the products and sums in the order of the definition.  fp64-bound: 4 slices of
// 169 x 3407 to 512 x 512 took 2.0 ms a pass with 12 taps per pixel, a twentieth so.
constexpr int kLJ = 64, kLI = 64, kLR = 192;  // columns, most rows of output, most plane rows
constexpr size_t kLSmem = ((size_t)kLR * kLJ + 8 * (kLI + kLJ)) * sizeof(double) + (kLI + kLJ) * sizeof(int);
template <int PASS>
__global__ void __launch_bounds__(kGT)
k_grid_lanczos(const int32_t* __restrict__ X, int h, int64_t nout, int64_t ns, int s0, int M, int ti, unsigned iruns,
               unsigned jruns, long long* __restrict__ work, uint8_t* __restrict__ out)
{
    extern __shared__ double sm[];
    double* H = sm;                      // [kLR][kLJ]
    double* wr = H + kLR * kLJ;          // [kLI][8]
    double* wc = wr + 8 * kLI;           // [kLJ][8]
    int* r0 = (int*)(wc + 8 * kLJ);      // [kLI]
    int* q0 = r0 + kLI;                  // [kLJ]
    const unsigned blk = PASS == 0 ? blockIdx.x : gridDim.x - 1 - blockIdx.x;
    const int j0 = (int)(blk % jruns) * kLJ, i0 = (int)(blk / jruns % iruns) * ti;
    const int s = s0 + (int)(blk / jruns / iruns);
    const int64_t c0 = (int64_t)s * ns;
    const int w = (int)min(ns, nout - c0);
    const int ni = min(ti, M - i0), nj = min(kLJ, M - j0);
    for (int e = (int)threadIdx.x; e < ni + nj; e += kGT) {
        double t[8];
        const bool row = e < ni;
        const int k = row ? lanczos_taps(i0 + e, h, M, t) : lanczos_taps(j0 + e - ni, w, M, t);
        double* to = row ? wr + 8 * e : wc + 8 * (e - ni);
#pragma unroll
        for (int a = 0; a < 8; a++) to[a] = t[a];
        if (row) r0[e] = k;
        else q0[e - ni] = k;
    }
    __syncthreads();
    const int jj = (int)threadIdx.x % kLJ, g = (int)threadIdx.x / kLJ;
    const int rb = r0[0], nr = r0[ni - 1] + 8 - rb;  // plane rows rb .. rb + nr - 1 (clamped to the plane)
    if (jj < nj) {
        double t[8];
        int q[8];
#pragma unroll
        for (int b = 0; b < 8; b++) {
            t[b] = wc[8 * jj + b];
            q[b] = min(max(q0[jj] + b, 0), w - 1);
        }
        for (int r = g; r < nr; r += kGT / kLJ) {
            const int32_t* x = X + (int64_t)min(max(rb + r, 0), h - 1) * nout + c0;
            double row = 0.0;
#pragma unroll
            for (int b = 0; b < 8; b++) row = fma(t[b], (double)__ldg(x + q[b]), row);
            H[r * kLJ + jj] = row;
        }
    }
    __syncthreads();
    long long lo = LLONG_MAX, hi = LLONG_MIN;
    const double ulo = PASS == 1 ? dval(work[2 * s]) : 0.0, uhi = PASS == 1 ? dval(work[2 * s + 1]) : 0.0;
    if (jj < nj)
        for (int i = g; i < ni; i += kGT / kLJ) {
            const double* Hr = H + (r0[i] - rb) * kLJ + jj;
            double U = 0.0;
#pragma unroll
            for (int a = 0; a < 8; a++) U = fma(wr[8 * i + a], Hr[a * kLJ], U);
            if (PASS == 0) {
                lo = min(lo, dkey(U));
                hi = max(hi, dkey(U));
            } else {
                out[((int64_t)s * M + i0 + i) * M + j0 + jj] =
                    (uint8_t)floor(255.0 * (U - ulo) / (uhi - ulo + 1e-6) + 0.5);
            }
        }
    if (PASS == 0) slice_minmax(lo, hi, work + 2 * s);
}

// Area path: pixel by pixel, or by columns.  Pixel / column time on planes of 60,000 at most, by the pixel's height x width in
// samples: M = 256: 1 x 1 0.52, 1 x 12 0.57, 1 x 20 0.76, 2 x 12 0.71, 2 x 20 0.98, 4 x 6 0.72, 4 x 20 1.2, 8 x 3 0.97; M = 64: 1 x 1
// 0.14, 2 x 20 0.51, 8 x 6 0.41, 8 x 20 0.96, 1 x 40 0.84; M = 2: all below 0.7.  (By columns lanes read consecutive samples; by
// pixels they read w / M apart, and rows of a few pixels leave no block half idle.)
bool by_pixel(int h, int64_t w, int M)
{
    const double a = (double)h * (double)w / ((double)M * M);  // samples of a pixel
    return M <= 32 ? a <= 300.0
                   : w <= 24 * (int64_t)M && (M < 256 ? a <= (M < 128 ? 100.0 : 56.0) : a <= 28.0 && h <= 6 * (int64_t)M);
}

// One pass over slices s0 .. s0 + n - 1, all on one path, in launches of as many
// slices as a grid holds.
int launch_pass(int pass, bool area, int n, cudaStream_t st, const int32_t* X, int h, int64_t nout, int64_t ns, int s0,
                int M, long long* work, uint8_t* out)
{
    const int64_t w = ns < nout - (int64_t)s0 * ns ? ns : nout - (int64_t)s0 * ns;
    const bool pixel = area && by_pixel(h, w, M);
    // area by columns: runs of kGT output columns of one row, with the columns they cover in shared memory
    const int64_t span = (std::min(M, kGT) * w + M - 1) / M + 1;
    const int cols = (int)std::max<int64_t>(2, (std::min<int64_t>(span, kGCBytes / 4) + 1) & ~1);
    // Lanczos: rows per block, as many as their plane rows fit (one row needs 8)
    const int ti = (int)std::max<int64_t>(1, std::min<int64_t>(kLI, (int64_t)(kLR - 9) * M / h));
    const unsigned iruns = (unsigned)((M + ti - 1) / ti), jruns = (unsigned)((M + kLJ - 1) / kLJ);
    const unsigned runs = (unsigned)(((pixel ? M * M : M) + kGT - 1) / kGT);
    const unsigned each = pixel ? runs : area ? (unsigned)M * runs : iruns * jruns;  // blocks of a slice
    if (!area)
        if (int rc = af_ensure_smem(pass == 0 ? (const void*)k_grid_lanczos<0> : (const void*)k_grid_lanczos<1>, kLSmem))
            return rc;
    for (int at = 0, per = (int)(0x7fffffffu / each); at < n; at += per) {
        const unsigned blocks = (unsigned)std::min(per, n - at) * each;
        const int s = s0 + at;
        if (pixel) {
            if (pass == 0) k_grid_pixel<0><<<blocks, kGT, 0, st>>>(X, h, nout, ns, s, M, runs, work, out);
            else k_grid_pixel<1><<<blocks, kGT, 0, st>>>(X, h, nout, ns, s, M, runs, work, out);
        } else if (area) {
            const size_t smem = (size_t)cols * 4;
            if (pass == 0) k_grid_area<0><<<blocks, kGT, smem, st>>>(X, h, nout, ns, s, M, runs, cols, work, out);
            else k_grid_area<1><<<blocks, kGT, smem, st>>>(X, h, nout, ns, s, M, runs, cols, work, out);
        } else {
            if (pass == 0) k_grid_lanczos<0><<<blocks, kGT, kLSmem, st>>>(X, h, nout, ns, s, M, ti, iruns, jruns, work, out);
            else k_grid_lanczos<1><<<blocks, kGT, kLSmem, st>>>(X, h, nout, ns, s, M, ti, iruns, jruns, work, out);
        }
        if (int rc = af_cuda_check(cudaGetLastError(), "af_grid launch")) return rc;
    }
    return AF_OK;
}

}  // namespace

extern "C" int af_grid(const int32_t* d_plane, int ndm, int64_t nout, int64_t ns, int M, uint8_t* d_out,
                       int64_t* d_work, void* stream)
try {
    if (!d_plane || !d_out || !d_work) return af_set_error(AF_EINVAL, "af_grid: NULL buffer");
    if (ndm < 1 || nout < 1 || ns < 1) return af_set_error(AF_EINVAL, "af_grid: empty plane or slice");
    if (M < 2 || M > 4096) return af_set_error(AF_EINVAL, "af_grid: M %d not in 2..4096", M);
    if (ns > INT32_MAX) return af_set_error(AF_EINVAL, "af_grid: slice too long");
    // exact area sums: |W| <= ndm * ns * 2^31 must stay below 2^63
    if ((double)ndm * (double)ns * 2147483648.0 >= 9.2e18)
        return af_set_error(AF_EINVAL, "af_grid: slices of %d x %lld values are too large for exact 64-bit sums", ndm,
                            (long long)ns);
    const int64_t S = (nout + ns - 1) / ns;
    if (S * M > 0x7fffffffLL) return af_set_error(AF_EINVAL, "af_grid: too many slices");
    cudaStream_t st = (cudaStream_t)stream;
    long long* work = reinterpret_cast<long long*>(d_work);
    k_grid_init<<<(unsigned)((S + 255) / 256), 256, 0, st>>>(work, (int)S);
    if (int rc = af_cuda_check(cudaGetLastError(), "af_grid init")) return rc;
    // full slices share one path; a shorter last slice may take the other
    const int64_t nfull = nout / ns;
    const int64_t last_w = nout - nfull * ns;
    const bool area_full = ndm > M && ns > M;
    const bool area_last = ndm > M && last_w > M;
    for (int pass = 0; pass < 2; pass++) {
        const bool one = nfull > 0 && last_w > 0 && area_full == area_last;  // every slice in one launch
        if (nfull > 0)
            if (int rc = launch_pass(pass, area_full, (int)(one ? S : nfull), st, d_plane, ndm, nout, ns, 0, M, work, d_out))
                return rc;
        if (last_w > 0 && !one)
            if (int rc = launch_pass(pass, area_last, 1, st, d_plane, ndm, nout, ns, (int)nfull, M, work, d_out)) return rc;
    }
    return AF_OK;
} catch (...) {
    return af_host_exception("af_grid");
}
