// cutout.cu -- the classifier's input: two 64 x 64 cut-outs around each
// candidate (DM-time from the plane, frequency-time from the input
// dedispersed at the candidate's DM), min-max normalised and rounded to
// bfloat16.  This replaces the paper's gridding of DM-time slices into
// 512 x 512 images (Sec. 2.4) and keeps its per-image min-max normalisation
// (without the 8-bit quantisation).  Definitions, per candidate (d, t, w):
//   bins       b = max(1, w / 2); bin j covers output samples
//              [t - 32 b + j b, t - 32 b + (j + 1) b), samples outside [0, nout) count 0
//   DM-time    [i][j] = sum over the bin of plane row d - 32 + i (0 outside [0, ndm))
//   freq-time  [g][j] = sum over channels c of group g (nchan / 64 each) and the
//              bin's samples s of X[c][s + D[d][c]]
//   normalise  v' = float(v - min) / (float(max - min) + 1e-6f), then bf16 (rn)
// Output NHWC bf16 [n][64][64][2]: channel 0 DM-time, 1 freq-time.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <limits.h>
#include <stdint.h>

#include "internal.h"
#include "nn.h"
#include "tile.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int S = 64;
constexpr int kCl = 8;                 // CTAs per candidate (one thread-block cluster)
constexpr int T = 256, NWARP = T / 32; // threads per CTA; warp w of CTA r owns image rows 8 r + w of both images
constexpr int CH = 512;                // DM-time: window positions per chunk, 16 per lane
constexpr int CHF = 508;               // frequency-time: positions per chunk (the last word's bytes shift out)
constexpr int kG = 4;                   // channels whose loads are issued together
constexpr int kDelaysInShared = 8192 / kCl;  // a CTA's channels whose delays are staged in shared memory
constexpr int kSortMax = 1024;         // candidates up to which clusters may take them widest first
constexpr int kRow = CH / 16 * 20;     // staged chunk: 16 positions every 20 words (no bank conflicts)

// Adds the column sums of window positions q0 .. q0 + 15 (q0 = the lane's first
// position, st = the warp's staged chunk) into the warp's 64 bins (bin j =
// positions [j b, (j+1) b); positions from 64 b on belong to no bin): one addition
// per bin the lane's positions touch.  A bin is two 32-bit words, sums of acc's low
// 20 bits and of the rest: 32-bit shared additions are one instruction, 64-bit ones
// a compare-and-swap loop that every lane of a wide bin takes part in.  fit: at
// most 2048 additions per bin, so neither word overflows; else the bin is one
// 64-bit word.  One copy of the code: the unrolled kernel otherwise misses its
// instruction cache.
__device__ __noinline__ void add_bins(const int32_t* st, int lane, int q0, int b, unsigned long long* wb, bool fit)
{
    int bin = q0 / b, edge = (bin + 1) * b;
    long long acc = 0;  // two's complement: plane values may be negative
    auto put = [&]() {
        if (bin < S && acc) {
            if (fit) {
                int* w = reinterpret_cast<int*>(wb + bin);
                atomicAdd(w, (int)(acc & 0xFFFFF));
                if (acc >> 20) atomicAdd(w + 1, (int)(acc >> 20));
            } else {
                atomicAdd(wb + bin, (unsigned long long)acc);
            }
        }
    };
#pragma unroll
    for (int q = 0; q < 4; q++) {
        const int4 u4 = *reinterpret_cast<const int4*>(st + lane * 20 + 4 * q);
        const int u[4] = {u4.x, u4.y, u4.z, u4.w};
#pragma unroll
        for (int jj = 0; jj < 4; jj++) {
            if (q0 + 4 * q + jj == edge) {  // entering the next bin
                put();
                acc = 0;
                bin++;
                edge += b;
            }
            acc += u[jj];
        }
    }
    put();
}

// One channel's words into the sums of bucket Q.  The comment keeps the compiler
// from merging the four into one indexed access (which puts the sums in memory).
template <int Q>
__device__ __forceinline__ void add_bucket(uint32_t (&A)[4][4], uint32_t (&O)[4][4], const uint32_t (&w)[4])
{
    asm volatile("// bucket %0" ::"n"(Q));
#pragma unroll
    for (int m = 0; m < 4; m++) {
        A[Q][m] += w[m];
        O[Q][m] += __byte_perm(w[m], 0u, 0x4341);
    }
}

// One channel's words into the sums of the bucket of its byte offset sh (the
// same in every lane).
__device__ __forceinline__ void add_words(uint32_t (&A)[4][4], uint32_t (&O)[4][4], const uint32_t (&w)[4], int sh)
{
    if (sh & 2) {
        if (sh & 1) add_bucket<3>(A, O, w);
        else add_bucket<2>(A, O, w);
    } else {
        if (sh & 1) add_bucket<1>(A, O, w);
        else add_bucket<0>(A, O, w);
    }
}

// Adds nc channels' words: channel k's window starts at x + k * nsamp + dl[k],
// x including the lane's 4 * lane bytes.  INNER: every word lies inside the input;
// else those outside its whole words first .. last read as 0.
template <bool INNER>
__device__ __forceinline__ void add_channels(uint32_t (&A)[4][4], uint32_t (&O)[4][4], const uint8_t* x, int64_t nsamp,
                                             const int32_t* dl, int nc, const uint8_t* first, const uint8_t* last)
{
    auto load = [&](uint32_t (&w)[4], int dc) {
        const uint8_t* a = x + dc;
        const int sh = (int)((uintptr_t)a & 3);
        a -= sh;
#pragma unroll
        for (int m = 0; m < 4; m++) {
            const uint8_t* am = a + 128 * m;
            w[m] = INNER || (am >= first && am <= last) ? __ldg(reinterpret_cast<const uint32_t*>(am)) : 0u;
        }
        x += nsamp;
        return sh;
    };
    int c = 0;
#pragma unroll 1
    for (; c + kG <= nc; c += kG) {
        uint32_t w[kG][4];
        int sh[kG];
#pragma unroll
        for (int k = 0; k < kG; k++) sh[k] = load(w[k], dl[c + k]);
#pragma unroll
        for (int k = 0; k < kG; k++) add_words(A, O, w[k], sh[k]);
    }
#pragma unroll 1
    for (; c < nc; c++) {
        uint32_t w[4];
        const int sh = load(w, dl[c]);
        add_words(A, O, w, sh);
    }
}

// Position of window position q of a chunk in the staged chunk.
__device__ __forceinline__ int staged(int q) { return q + (q >> 4) * 4; }

// An input that starts mis bytes after a 4-byte address: adds its bytes outside the
// whole words (the first 4 - mis, of channel 0, and the last mis, of the last
// channel) into the staged chunk of channels c .. c + nc - 1 (delays dl), n
// positions from sample s0 on.
__device__ __noinline__ void add_ends(int32_t* st, int lane, const uint8_t* X, int64_t nsamp, int nchan, int mis, int c,
                                      int nc, const int32_t* dl, int64_t s0, int n, int64_t nout)
{
    const bool head = lane < 4 - mis && c == 0, tail = lane >= 4 - mis && lane < 4 && c + nc == nchan;
    if (head || tail) {
        const int64_t at = head ? lane : nsamp - 4 + lane;  // sample of its channel
        const int64_t q = at - dl[head ? 0 : nc - 1] - s0;
        if (q >= 0 && q < n && s0 + q >= 0 && s0 + q < nout)
            st[staged((int)q)] += __ldg(X + (int64_t)(head ? 0 : nchan - 1) * nsamp + at);
    }
    __syncwarp();
}

// The candidate of rank `rank` when all n <= kSortMax are taken widest first (by
// the widths' binary order of magnitude, then by index).  mask: kSortMax / 32 rows of
// 32 words.  Every thread of the CTA calls it.
__device__ int ranked(const af_cand_t* __restrict__ cands, int n, int rank, uint32_t* mask, int* found)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, chunks = (n + 31) / 32;
    // which of every 32 candidates are in which class: mask[32 c + class], one ballot per class there
    constexpr int PER = kSortMax / 32 / NWARP;
    int cls[PER];
#pragma unroll
    for (int k = 0; k < PER; k++) {
        const int i = 32 * (warp + k * NWARP) + lane;
        cls[k] = i < n ? __clz(max(1, __ldg(&cands[i].width))) : 32;  // small for wide
    }
#pragma unroll
    for (int k = 0; k < PER; k++) {
        const int c = warp + k * NWARP;
        if (c >= chunks) break;  // the same in every lane
        mask[32 * c + lane] = 0u;
        __syncwarp();  // the clear comes before the store
        const uint32_t m = __match_any_sync(0xffffffffu, cls[k]);
        if (cls[k] < 32 && lane == __ffs(m) - 1) mask[32 * c + cls[k]] = m;
    }
    __syncthreads();
    if (warp == 0) {
        // what lane `at` of the warp holds when the lanes' counts pass `left`; left becomes the rest
        auto pass = [&](int cnt, int& left) {
            int incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            const int at = __ffs(__ballot_sync(0xffffffffu, left < incl)) - 1;
            left -= __shfl_sync(0xffffffffu, incl - cnt, at);
            return at;
        };
        int left = rank, tot = 0;
        for (int c = 0; c < chunks; c++) tot += __popc(mask[32 * c + lane]);
        const int k = pass(tot, left);                                            // the class
        const int c = pass(lane < chunks ? __popc(mask[32 * lane + k]) : 0, left);  // its 32 candidates
        const int b = pass((int)(mask[32 * c + k] >> lane & 1u), left);             // its bit
        if (lane == 0) *found = 32 * c + b;
    }
    __syncthreads();
    return *found;
}

// One cluster of kCl CTAs per candidate; CTA r computes DM-time rows and
// frequency-time rows 8 r .. 8 r + 7, warp w of it row 8 r + w of each image.
// Window positions q in [0, 64 b) are samples start + q, start = t - 32 b;
// samples outside [0, nout) count 0.  A warp walks its rows in chunks, lane l
// holding positions 16 l .. 16 l + 15 of the chunk (512 positions for the
// DM-time row, 508 for the frequency-time row).  DM-time values are loaded 32
// consecutive at a time and staged in shared memory.  The frequency-time row adds
// its channels as the dedispersion tile kernel does: aligned 32-bit words (four per
// lane and channel, kG channels' loads issued together), bucketed by the byte the
// window starts at, A += w and O += the odd bytes, the buckets folded once per
// chunk; positions that do not count are cleared after the fold.  Then the chunk
// is added into the warp's bins.  The images' minimum and maximum are reduced over the cluster through
// distributed shared memory; every CTA of a cluster takes the same path (one
// candidate), so both cluster barriers are reached by all of them.
// Bound by the loads' latency.  256 candidates of widths 1 to 256, 4096 channels,
// cut out and classified: 477 us (880 to 920 with 16-byte loads realigned by shuffles
// and masked per channel, 64-bit bins and plane values loaded 64 bytes apart);
// 3 CTAs per SM with 4 channels in flight a warp: 473, 2 with 8: 479, 4 with 2: 539.
// Inputs at any byte address (1024 channels, rows off a 4-byte address, 64 candidates
// of width 16: 93 us byte by byte, 33 so).
// Clusters take the widest candidates of a list of moderate length first, so that no
// long one starts last: in the list's order 625 us.
__global__ void __cluster_dims__(kCl, 1, 1) __launch_bounds__(T, 3)
k_cutout(const uint8_t* __restrict__ X, int64_t nsamp, int nchan, const int32_t* __restrict__ D, int ndm,
         const int32_t* __restrict__ plane, int64_t nout, const af_cand_t* __restrict__ cands, int n, bool order,
         __nv_bfloat16* __restrict__ out)
{
    __shared__ unsigned long long wbins[NWARP][2][S];  // per warp: bins of its DM-time and frequency-time rows
    __shared__ int32_t sD[kDelaysInShared];            // the delays of this CTA's channels (when they fit)
    __shared__ long long red[NWARP][4];                // per-warp min / max of both images
    __shared__ __align__(16) int32_t stage[NWARP][kRow];  // first: the ranking's masks
    static_assert(kSortMax <= 1024 && sizeof(int32_t) * NWARP * kRow >= kSortMax * 4, "masks of 32 rows of 32 words");
    __shared__ int found;
    __shared__ long long mm[4];                        // this CTA's: DM-time min, max, frequency-time min, max
    cg::cluster_group cluster = cg::this_cluster();
    const int r = (int)cluster.block_rank();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cand = order ? ranked(cands, n, (int)(blockIdx.x / kCl), reinterpret_cast<uint32_t*>(stage), &found)
                           : (int)(blockIdx.x / kCl);
    const af_cand_t cd = cands[cand];
    const int d = cd.dm_idx;
    __nv_bfloat16* o = out + (int64_t)cand * S * S * 2;
    const int row = NWARP * r + warp;  // image row of this warp (both images)
    if (d < 0 || d >= ndm) {  // not a row of this plan: zero cut-outs (the whole cluster returns here)
        for (int e = threadIdx.x; e < NWARP * S * 2; e += T) o[NWARP * r * S * 2 + e] = __float2bfloat16(0.f);
        return;
    }
    const int b = cd.width / 2 > 1 ? cd.width / 2 : 1;
    const int64_t start = (int64_t)cd.t - 32 * (int64_t)b;
    const int span = S * b;
    const int gsz = nchan / S;
    const int cb = NWARP * r * gsz, ce = cb + NWARP * gsz;  // this CTA's channels
    const bool dsh = ce - cb <= kDelaysInShared;
    if (dsh)
        for (int c = cb + threadIdx.x; c < ce; c += T) sD[c - cb] = __ldg(D + (int64_t)d * nchan + c);
    for (int e = lane; e < 2 * S; e += 32) (&wbins[warp][0][0])[e] = 0ull;
    __syncthreads();

    // the bins' two 32-bit words hold every sum
    const bool fit = b <= 2048 && (int64_t)gsz * 255 * b < (int64_t)1 << 31;
    int32_t* st = stage[warp];
    // DM-time row: plane row d - 32 + row (0 outside the plan)
    const int pr = d - 32 + row;
    if (pr >= 0 && pr < ndm) {
        const int32_t* yr = plane + (int64_t)pr * nout;
        for (int p0 = 0; p0 < span; p0 += CH) {
            if (start + p0 + CH <= 0 || start + p0 >= nout) continue;  // no position counts
#pragma unroll
            for (int jj = 0; jj < CH / 32; jj++) {
                const int q = p0 + 32 * jj + lane;
                const int64_t sm = start + q;
                st[staged(32 * jj + lane)] = q < span && sm >= 0 && sm < nout ? __ldg(yr + sm) : 0;
            }
            __syncwarp();
            add_bins(st, lane, p0 + 16 * lane, b, wbins[warp][0], fit);
            __syncwarp();
        }
    }
    // frequency-time row: channels row * gsz .. (row + 1) * gsz
    // the input's first and last whole word; at a 4-byte address they hold all of it (nchan is a multiple of 64)
    const int mis = (int)(reinterpret_cast<uintptr_t>(X) & 3);
    const uint8_t* const first = X + (4 - mis) % 4;
    const uint8_t* const last = X + (int64_t)nchan * nsamp - 4 - mis;
    const int32_t* dl = dsh ? sD + (row * gsz - cb) : D + (int64_t)d * nchan + row * gsz;  // the row's delays
    for (int p0 = 0; p0 < span; p0 += CHF) {
        const int64_t s0 = start + p0;  // sample of the chunk's first position
        if (s0 + CHF <= 0 || s0 >= nout) continue;  // no position counts
        const bool inner = s0 >= 3 && s0 + CH <= nout;  // every word of every channel lies inside its row
        const bool full = s0 >= 0 && s0 + CHF <= nout && p0 + CHF <= span;  // every position counts
        for (int c0 = 0; c0 < gsz; c0 += 256) {  // 16-bit lanes hold 256 channels
            const int nc = min(256, gsz - c0);
            const uint8_t* x = X + (int64_t)(row * gsz + c0) * nsamp + s0;
            uint32_t u[4][4];  // column sums of positions 4 (lane + 32 m) + k, at most 255 * 256
            uint32_t A[4][4], O[4][4];
#pragma unroll
            for (int q = 0; q < 4; q++)
#pragma unroll
                for (int m = 0; m < 4; m++) A[q][m] = O[q][m] = 0u;
            if (inner) add_channels<true>(A, O, x + 4 * lane, nsamp, dl + c0, nc, first, last);
            else add_channels<false>(A, O, x + 4 * lane, nsamp, dl + c0, nc, first, last);
#pragma unroll
            for (int m = 0; m < 4; m++)
#pragma unroll
                for (int k = 0; k < 4; k++) u[m][k] = 0u;
            aftile::Tile<1, 4>::fold(A, O, u, lane);
#pragma unroll
            for (int m = 0; m < 4; m++) {
                const int p = 4 * (lane + 32 * m);
                if (!full) {
#pragma unroll
                    for (int k = 0; k < 4; k++)
                        if (p + k >= CHF || p0 + p + k >= span || s0 + p + k < 0 || s0 + p + k >= nout) u[m][k] = 0u;
                } else if (p >= CHF) {
                    u[m][0] = u[m][1] = u[m][2] = u[m][3] = 0u;
                }
                *reinterpret_cast<uint4*>(st + staged(p)) = make_uint4(u[m][0], u[m][1], u[m][2], u[m][3]);
            }
            __syncwarp();
            if (mis && !inner) add_ends(st, lane, X, nsamp, nchan, mis, row * gsz + c0, nc, dl + c0, s0, min(CHF, span - p0), nout);
            add_bins(st, lane, p0 + 16 * lane, b, wbins[warp][1], fit);
            __syncwarp();
        }
    }
    __syncwarp();
    long long bins[2][2];  // [DM-time, frequency-time][column 2 lane + h]
#pragma unroll
    for (int k = 0; k < 2; k++) {
        for (int h = 0; h < 2; h++) {
            const long long w = (long long)wbins[warp][k][2 * lane + h];
            bins[k][h] = fit ? ((w >> 32) << 20) + (long long)(uint32_t)w : w;
        }
    }

    // min / max of both images: warp, CTA, then the cluster (distributed shared memory)
    long long v[4] = {min(bins[0][0], bins[0][1]), max(bins[0][0], bins[0][1]), min(bins[1][0], bins[1][1]),
                      max(bins[1][0], bins[1][1])};
#pragma unroll
    for (int o2 = 16; o2 > 0; o2 >>= 1) {
        v[0] = min(v[0], __shfl_xor_sync(0xffffffffu, v[0], o2));
        v[1] = max(v[1], __shfl_xor_sync(0xffffffffu, v[1], o2));
        v[2] = min(v[2], __shfl_xor_sync(0xffffffffu, v[2], o2));
        v[3] = max(v[3], __shfl_xor_sync(0xffffffffu, v[3], o2));
    }
    if (lane == 0)
        for (int i = 0; i < 4; i++) red[warp][i] = v[i];
    __syncthreads();
    if (threadIdx.x == 0) {
        long long m[4] = {LLONG_MAX, LLONG_MIN, LLONG_MAX, LLONG_MIN};
        for (int w = 0; w < NWARP; w++) {
            m[0] = min(m[0], red[w][0]);
            m[1] = max(m[1], red[w][1]);
            m[2] = min(m[2], red[w][2]);
            m[3] = max(m[3], red[w][3]);
        }
        for (int i = 0; i < 4; i++) mm[i] = m[i];
    }
    cluster.sync();  // every CTA's mm is written
    long long g[4] = {LLONG_MAX, LLONG_MIN, LLONG_MAX, LLONG_MIN};
    for (int q = 0; q < kCl; q++) {
        const long long* rm = cluster.map_shared_rank(mm, q);
        g[0] = min(g[0], rm[0]);
        g[1] = max(g[1], rm[1]);
        g[2] = min(g[2], rm[2]);
        g[3] = max(g[3], rm[3]);
    }
    cluster.sync();  // no CTA leaves while another may still read its mm
    const float ad = (float)(g[1] - g[0]) + 1e-6f, fd = (float)(g[3] - g[2]) + 1e-6f;
#pragma unroll
    for (int k = 0; k < 2; k++) {
        const bool ft = k == 1;
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int e = row * S + 2 * lane + h;
            const float x = ft ? __fdiv_rn((float)(bins[k][h] - g[2]), fd) : __fdiv_rn((float)(bins[k][h] - g[0]), ad);
            o[2 * e + (ft ? 1 : 0)] = __float2bfloat16_rn(x);
        }
    }
}

}  // namespace

int nn_cutouts(const uint8_t* X, int64_t nsamp, int nchan, const int32_t* D, int ndm, const int32_t* plane,
               int64_t nout, const af_cand_t* cands, int n, __nv_bfloat16* out, cudaStream_t s)
{
    if (n <= 0) return AF_OK;
    if ((long long)n * kCl > 0x7fffffffLL) return af_set_error(AF_EINVAL, "cut-outs: too many candidates for one grid");
    // Widest first pays where one wide candidate would start last, and costs every block a look at the whole list: worth
    // it up to about 9 waves of clusters (57 of them run at a time), twice that where a candidate's own work is longer.
    // 512 candidates, ordered / not: widths mixed 1 to 256, 4096 channels 805 / 945 us, 64 channels 238 / 242; width 1, 64
    // channels 130 / 115; 1024 at 4096 channels 1605 / 1772; 4000, every block ranking all (before): 7264 / 6340.
    const bool order = n > 8 && n <= (nchan >= 512 ? kSortMax : kSortMax / 2);
    k_cutout<<<(unsigned)n * kCl, T, 0, s>>>(X, nsamp, nchan, D, ndm, plane, nout, cands, n, order, out);
    return af_cuda_check(cudaGetLastError(), "cut-out launch");
}
