// pairs.cu -- exact brute-force dedispersion (Sec. 2.3) of single plans
// through shared channel-group rows.
//
//   Y[d][t] = sum_c X[c][t + D[d][c]]
//           = sum_q P(q, delta_q(d))[t + D[d][Gq]],
//   P(q, delta)[u]   = sum_{i<G} X[Gq+i][u + delta_i],  delta_0 = 0,
//   delta_q(d)_i     = D[d][Gq+i] - D[d][Gq],
//
// for groups of G = 2, 3 or 4 adjacent channels (a short last group has zeros
// for its missing channels).  The same integer sum, grouped: the channels of
// a group are added once per distinct tuple of relative delays (a group has a
// few dozen over the whole DM range and a few inside a block of neighbouring
// DMs), and the DM sums then run over group rows, nchan / G terms.
//
// Stage 1 (k_group_rows<G>) writes every row P(q, delta) as uint16 for one
// time block of L outputs; row g covers only the delays D[d][Gq] of the DMs
// that use it (element e is time T0 + B_g + e, B_g their smallest delay
// rounded down to 16).
//
// Stage 2 (k_pair_tile) is a tile kernel over rows: a block takes 15 or 30 DM
// rows (15 consumer warps with one or two DMs each, DMs ascending) and TTE = 1016
// outputs; a producer warp streams the block's row windows (one per block and
// row) through an NS-deep shared-memory ring, up to 32 windows of whole groups
// packed back to back per stage, one bulk async copy per window plus one for the
// chunk's consumer tables of (window, offset) per group, which the host computes
// once (tiles start at multiples of 8, so no offset depends on the tile).  Lane L
// of a consumer warp owns outputs 2 (L + 32 m) + k, m < 16, k < 2, of each of its
// DMs: one aligned 32-bit shared load brings the two 16-bit samples of a group, so
// the groups are bucketed by the parity r of the sample offset; one IADD3 adds two
// rows' words into the 16-bit lanes of the bucket's accumulator (at most
// 65535 / (255 G) rows between folds); a fold re-aligns bucket 1 by one sample (one
// lane shuffle) into the 32-bit output sums.
//
// What bounds stage 2: the consumers' shared loads (2 bytes per DM, group and
// output) and the window copies from L2 (7.6 TB/s on GB300), which take as long
// as each other with 15 DM rows per block (4096 channels, 1001 DMs, 215,261
// outputs, groups of 3: 17.0 ms each alone, 19.2 ms together).  A block of 30 rows
// copies 0.68 of the bytes per output, since neighbouring DMs share rows; its
// bucket accumulators fill the registers that 15 rows' accumulators and 32-bit
// sums took, and the 32-bit sums, touched once per fold, live in tensor memory
// (which no other part of this kernel uses): 17.2 ms with groups of 3, and groups
// of 4, whose loads take 13.2 ms alone, 18.8 -> 14.3 ms.
//
// Every wait is bounded (the tile kernel's error flag).  The host tables of
// every group size and block height are built once per plan; a reservation picks
// one by a cost model, uploads it and sizes the row buffer from a budget.
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdlib.h>

#include <algorithm>
#include <array>
#include <cmath>
#include <future>
#include <numeric>
#include <type_traits>
#include <vector>

#include "internal.h"
#include "ptx.cuh"
#include "umma.cuh"

namespace {

constexpr int kPNW = 15;            // consumer warps per block, each with 1 or 2 DM rows (DPW)
// Ring: up to kPSL row windows per stage (one per producer lane), packed back
// to back (a stage holds as many whole groups as fit its bytes); the depth is
// 2, 3 or 4 stages (AFGB_PAIR_STAGES at plan creation, default 3: on the
// 4096-channel workload with groups of 3, stage 2 took 19.8 / 19.2 / 21.5 ms).
constexpr int kPSL = 32;
constexpr int kPMG = 16;            // 2-sample groups per lane
constexpr int kPTTE = 1016;         // outputs per tile: a multiple of 8 below 64 * kPMG - 1
constexpr int kPTABW = 40;          // uint16 per (stage, DM row) table: 2 starts, 2 counts, <= 34 offsets / 4
constexpr int kPTM = 256;           // tensor-memory columns of a block (DPW = 2)
constexpr uint32_t kPWait = afptx::kMbarWaitPolls;
constexpr int kET = 4096;           // stage 1: row samples per block
constexpr int kS1T = 256;
constexpr int kMaxDr = 32768;       // stage 1: largest range of one relative delay over a group's rows
constexpr int kMinTiles = 8;        // smallest useful time block, in tiles

inline int64_t r8(int64_t x) { return (x + 7) & ~(int64_t)7; }
inline int64_t r16(int64_t x) { return (x + 15) & ~(int64_t)15; }

typedef af_pair_args PairArgs;

// ------------------------------------------------------------------ stage 1
// Block = (group q of G channels, ET samples of the group's range); writes,
// for every row of the group, the part of those samples inside the row's own
// range.  pinfo[q] = {first row, rows, ub (the group's first delay rounded down
// to 16), length of the group's range}; rinfo[g] = {row start - ub (a multiple
// of 16), row length}; rdelta[g][i-1] = row g's delay of channel Gq+i relative
// to channel Gq; gdr[q][i-1] = the smallest and largest of those over the
// group's rows.  Channel Gq's window goes to W0, channel Gq+i's (shifted by
// the smallest delta, longer by the delta range + 4 bytes) to Wi: blocks whose
// windows lie inside the input rows copy them with aligned 16-byte loads (a
// window then starts off_i bytes into its buffer), edge blocks the same with
// zeros outside the rows and for missing channels (byte by byte a row's last
// block alone took 20 us).  Words at any byte
// offset are read with a funnel shift (one shift per block and row).
// A group's rows come in lexicographic order of their tuples, so that a row
// mostly shares its first delays with the one before: the sums over those
// channels stay in registers and only the channels from the first difference on
// are read and widened again (1.36 of 2 per row for groups of 3, 1.61 of 3 for
// groups of 4 on the 4096-channel workload).  Bound by HBM (groups of 4: 36.9 GB in
// 5.34 ms, its measured rate; every channel read again for every row: 6.64 ms, 15
// ALU instructions per 4 samples and row) or, where rows are few or short, by
// issue.  With every row waiting for its own record, and edge windows copied byte
// by byte, 3508 channels, 1287 DMs, 19024 outputs took 258 us in groups of 4, 137 so;
// 271 channels, 543 DMs, 22053 outputs 53 us, 25 so.  8 - G blocks per SM: one
// block more spills or is slower (G = 4: 1.00 to 1.27 ms), one less up to 1.13 times
// slower.
template <int G>
__global__ void __launch_bounds__(kS1T, 8 - G)
k_group_rows(const uint8_t* __restrict__ X, int64_t nsamp, int nchan, const int4* __restrict__ pinfo,
             const int2* __restrict__ gdr, const int32_t* __restrict__ rdelta,
             const int2* __restrict__ rinfo, const int64_t* __restrict__ rowoff, int64_t T0, int etiles, int wstride,
             int dshort, uint16_t* __restrict__ PS)
{
    constexpr int K = G - 1;
    extern __shared__ __align__(16) uint8_t sm[];
    __shared__ int64_t s_ro[kS1T];
    __shared__ int2 s_ri[kS1T];
    __shared__ int s_dl[K][kS1T];
    __shared__ int s_cnt[kS1T / 32];
    __shared__ uint8_t s_list[kS1T];
    const int tid = threadIdx.x;
    const int q = blockIdx.x / etiles;
    const int64_t e0 = (int64_t)(blockIdx.x % etiles) * kET;
    const int4 pi = __ldg(pinfo + q);
    // a time block dshort outputs shorter than the layout's needs every row
    // (and the group's range) dshort samples shorter (dshort a multiple of 16)
    if (e0 >= pi.w - dshort) return;
    // The records of the group's rows in shared memory, kS1T rows a pass, and the
    // list of those that overlap [e0, e0 + ET): one load per thread, instead of
    // every row's sum waiting for its own record.
    bool over = false;
    auto load_records = [&](int kb) {
        over = false;
        if (kb + tid < pi.y) {
            const int g = pi.x + kb + tid;
            const int2 r = __ldg(rinfo + g);
            s_ri[tid] = make_int2(r.x, r.y - dshort);
            s_ro[tid] = __ldg(rowoff + g);
#pragma unroll
            for (int i = 0; i < K; i++) s_dl[i][tid] = __ldg(rdelta + (int64_t)g * K + i);
            over = r.x < e0 + kET && r.x + r.y - dshort > e0;
        }
    };
    // ends with a barrier; returns the list's length
    auto list_records = [&]() {
        const unsigned bal = __ballot_sync(0xffffffffu, over);
        if ((tid & 31) == 0) s_cnt[tid >> 5] = __popc(bal);
        __syncthreads();
        int n = 0, at = 0;
#pragma unroll
        for (int w = 0; w < kS1T / 32; w++) {
            if (w == (tid >> 5)) at = n;
            n += s_cnt[w];
        }
        if (over) s_list[at + __popc(bal & ((1u << (tid & 31)) - 1u))] = (uint8_t)tid;
        __syncthreads();
        return n;
    };
    load_records(0);
    const int c0 = G * q;
    const int64_t u0 = T0 + pi.z + e0;
    int dmn[K], bw[K], off[K + 1];
    bool fast = u0 >= 0 && u0 + kET + 48 <= nsamp;
#pragma unroll
    for (int i = 0; i < K; i++) {
        const int2 r = __ldg(gdr + (int64_t)q * K + i);
        dmn[i] = r.x;
        bw[i] = kET + (r.y - r.x) + 4;  // + the word the last funnel shift reads past
        fast = fast && c0 + 1 + i < nchan && u0 + r.x >= 0 && u0 + r.x + bw[i] + 48 <= nsamp;
    }
    const uint8_t* x0 = X + (int64_t)c0 * nsamp + u0;
    if (fast) {
        off[0] = (int)((uintptr_t)x0 & 15);
        const uint4* g0 = reinterpret_cast<const uint4*>(x0 - off[0]);
        const int n0 = (off[0] + kET + 4 + 15) >> 4;
        for (int k = tid; k < n0; k += kS1T) reinterpret_cast<uint4*>(sm)[k] = __ldg(g0 + k);
#pragma unroll
        for (int i = 0; i < K; i++) {
            const uint8_t* xi = X + (int64_t)(c0 + 1 + i) * nsamp + u0 + dmn[i];
            off[i + 1] = (int)((uintptr_t)xi & 15);
            const uint4* gi = reinterpret_cast<const uint4*>(xi - off[i + 1]);
            uint4* wi = reinterpret_cast<uint4*>(sm + kET + 48 + i * wstride);
            const int ni = (off[i + 1] + bw[i] + 4 + 15) >> 4;
            for (int k = tid; k < ni; k += kS1T) wi[k] = __ldg(gi + k);
        }
    } else {
        // the same 16-byte pieces; those outside the row (or of a missing channel) are
        // zero, the one that straddles an end is copied byte by byte
        auto edge = [&](uint8_t* w, int c, int64_t u, int bytes) {
            const bool have = c < nchan;
            const uint8_t* x = X + (int64_t)(have ? c : c0) * nsamp + u;
            const int o = (int)((uintptr_t)x & 15);
            const int n = (o + bytes + 15) >> 4;
            for (int k = tid; k < n; k += kS1T) {
                const int64_t s = u - o + 16 * k;
                uint4 v = make_uint4(0u, 0u, 0u, 0u);
                if (have && s >= 0 && s + 16 <= nsamp) v = __ldg(reinterpret_cast<const uint4*>(x - o) + k);
                reinterpret_cast<uint4*>(w)[k] = v;
                if (have && s < nsamp && s + 16 > 0 && (s < 0 || s + 16 > nsamp))
                    for (int i = (int)max((int64_t)0, -s); i < (int)min((int64_t)16, nsamp - s); i++)
                        w[16 * k + i] = __ldg(x - o + 16 * k + i);
            }
            return o;
        };
        off[0] = edge(sm, c0, u0, kET + 4);
#pragma unroll
        for (int i = 0; i < K; i++) off[i + 1] = edge(sm + kET + 48 + i * wstride, c0 + 1 + i, u0 + dmn[i], bw[i] + 4);
    }
    int nrec = list_records();  // its barriers also complete the windows
    // thread tid takes the 4-sample words w = tid + 256 j (j < 4) of the block:
    // consecutive lanes read consecutive shared words (no bank conflicts) and
    // store consecutive 8-byte pieces of a row
    // sums over the group's first i + 1 channels at the current delays, two 16-bit lanes a word
    uint32_t lo[K][4], hi[K][4];
    bool live[4];
    {
        const uint32_t* A32 = reinterpret_cast<const uint32_t*>(sm);
        const uint32_t sh = (uint32_t)(off[0] & 3) * 8u;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int w = tid + kS1T * j;
            live[j] = e0 + 4 * w < pi.w - dshort;
            const int p = (off[0] >> 2) + w;
            const uint32_t a = __funnelshift_r(A32[p], A32[p + 1], sh);
            lo[0][j] = __byte_perm(a, 0u, 0x4140);  // samples 0, 1 into 16-bit lanes
            hi[0][j] = __byte_perm(a, 0u, 0x4342);  // samples 2, 3
        }
    }
    int prev[K];
#pragma unroll
    for (int i = 0; i < K; i++) prev[i] = INT32_MIN;
    for (int kb = 0, k = 0; kb < pi.y; k++) {
        if (k == nrec) {  // the same in every thread: the next pass
            kb += kS1T;
            k = -1;
            nrec = 0;
            if (kb < pi.y) {
                __syncthreads();  // every thread is done with the records before
                load_records(kb);
                nrec = list_records();
            }
            continue;
        }
        const int rec = s_list[k];
        const int start = s_ri[rec].x, len = s_ri[rec].y;
        uint16_t* row = PS + s_ro[rec];
        int d[K];
#pragma unroll
        for (int i = 0; i < K; i++) d[i] = s_dl[i][rec];
        bool change = false;  // a delay so far differs from the last summed row's (the same in every thread)
        uint32_t l[4], h[4];
#pragma unroll
        for (int i = 0; i < K; i++) {
            change = change || d[i] != prev[i];
            prev[i] = d[i];
            if (!change && i < K - 1) continue;
            const uint32_t* W32 = reinterpret_cast<const uint32_t*>(sm + kET + 48 + i * wstride);
            const int pb = off[i + 1] + d[i] - dmn[i];
            const uint32_t sh = (uint32_t)(pb & 3) * 8u;
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int p = (pb >> 2) + tid + kS1T * j;
                const uint32_t b = __funnelshift_r(W32[p], W32[p + 1], sh);
                l[j] = lo[i][j] + __byte_perm(b, 0u, 0x4140);
                h[j] = hi[i][j] + __byte_perm(b, 0u, 0x4342);
                if (i < K - 1) {
                    lo[i + 1 < K ? i + 1 : 0][j] = l[j];
                    hi[i + 1 < K ? i + 1 : 0][j] = h[j];
                }
            }
        }
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int rel = (int)e0 + 4 * (tid + kS1T * j) - start;  // sample index within the row
            if (live[j] && (uint32_t)rel < (uint32_t)len)
                *reinterpret_cast<uint2*>(row + rel) = make_uint2(l[j], h[j]);
        }
    }
}

// ------------------------------------------------------------------ stage 2
template <int NS, int DPW>
struct PairTile {
    static constexpr int NW = kPNW, ND = NW * DPW;      // consumer warps, DM rows of a block
    static constexpr uint32_t TB = ND * kPTABW * 2;     // table bytes of a chunk

    static __device__ __forceinline__ int2 load_cd(const PairArgs& a, int cbeg, int nchk, int kk)
    {
        return kk < nchk ? __ldg(a.chunks + cbeg + kk) : make_int2(0, 0);
    }

    // Chunk c (block-local kk) into stage st: its precomputed table block and
    // one window per row slot, all completing on the stage's full barrier.
    static __device__ __forceinline__ void produce(const PairArgs& a, uint8_t* smem, uint16_t* tab, uint32_t full_bar,
                                                   int c, const int2& cd, uint32_t bytes, uint32_t soff,
                                                   int64_t src, int st, int lane)
    {
        const uint32_t tot = __reduce_add_sync(0xffffffffu, bytes) + TB;
        __syncwarp();
        afptx::fence_proxy_async();  // the consumers' reads of this stage come before the copies
        if (lane == 0) {
            afptx::mbar_arrive_expect_tx(full_bar, tot);
            afptx::bulk_g2s(afptx::smem_addr(tab + st * ND * kPTABW), a.tabs + (int64_t)c * ND * kPTABW, TB, full_bar);
        }
        __syncwarp();
        if (lane < cd.x && bytes)
            afptx::bulk_g2s(afptx::smem_addr(smem) + (uint32_t)(st * a.stage_bytes + soff), a.PS + src, bytes,
                            full_bar);
    }

    // Adds half h (groups 8 h .. 8 h + 7) of the bucket accumulators into the
    // 32-bit sums w[2 (m - 8 h) + k] and clears them.  Bucket 1 holds, in lane L
    // group m, samples 2 (L + 32 m) + 1 and + 2: output k = 0 takes its own upper
    // half, k = 1 the lower half of the next lane's word (lane 0 of group m + 1 for
    // L = 31).  Halves in descending order: `carry` runs through both.
    static __device__ __forceinline__ void fold_half(uint32_t (&A)[2][kPMG], int h, uint32_t (&w)[kPMG], uint32_t& carry,
                                                     int lane)
    {
#pragma unroll
        for (int i = 7; i >= 0; i--) {
            const int m = 8 * h + i;
            const uint32_t a0 = A[0][m], a1 = A[1][m];
            const uint32_t lo1 = a1 & 0xFFFFu;
            uint32_t nx = __shfl_down_sync(0xffffffffu, lo1, 1);
            const uint32_t l0 = __shfl_sync(0xffffffffu, lo1, 0);
            if (lane == 31) nx = carry;
            carry = l0;
            w[2 * i] += (a0 & 0xFFFFu) + (a1 >> 16);
            w[2 * i + 1] += (a0 >> 16) + nx;
            A[0][m] = 0u;
            A[1][m] = 0u;
        }
    }

    // The 32-bit sums of a warp's DM rows: registers (one row), or tensor memory
    // (two rows: lanes 32 (warp % 4) .., 32 columns per row), read, added to and
    // written back 16 columns at a time.
    struct Sums {
        uint32_t r[DPW == 1 ? 2 : 1][kPMG];
        uint32_t taddr;
        __device__ __forceinline__ void init(uint32_t tmem, int warp)
        {
            if (DPW == 1) {
#pragma unroll
                for (int i = 0; i < kPMG; i++) r[0][i] = r[DPW == 1 ? 1 : 0][i] = 0u;
            } else {
                taddr = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(64 * (warp >> 2));
                uint32_t z[16];
#pragma unroll
                for (int i = 0; i < 16; i++) z[i] = 0u;
#pragma unroll
                for (int c = 0; c < 4; c++) afumma::st_32x32b_x16(taddr + 16 * c, z);
                afumma::wait_st();
            }
        }
        __device__ __forceinline__ void fold(uint32_t (&A)[2][kPMG], int u, int lane)
        {
            uint32_t carry = 0u;
#pragma unroll
            for (int h = 1; h >= 0; h--) {
                if (DPW == 1) {
                    fold_half(A, h, r[DPW == 1 ? h : 0], carry, lane);
                } else {
                    uint32_t w[16];
                    afumma::ld_32x32b_x16(taddr + 32 * u + 16 * h, w);
                    afumma::wait_ld();
                    fold_half(A, h, w, carry, lane);
                    afumma::st_32x32b_x16(taddr + 32 * u + 16 * h, w);
                }
            }
            if (DPW == 2) afumma::wait_st();
        }
        // half h of row u
        __device__ __forceinline__ void get(int u, int h, uint32_t (&w)[kPMG]) const
        {
            if (DPW == 1) {
#pragma unroll
                for (int i = 0; i < kPMG; i++) w[i] = r[DPW == 1 ? h : 0][i];
            } else {
                afumma::ld_32x32b_x16(taddr + 32 * u + 16 * h, w);
                afumma::wait_ld();
            }
        }
    };

    // DM block jb, outputs t0 .. t0 + TTE - 1 of the time block a.T0.
    static __device__ __forceinline__ void run(const PairArgs& a, uint8_t* smem, unsigned jb, int64_t t0, uint32_t tmem)
    {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        uint16_t* tab = (uint16_t*)(smem + (size_t)NS * a.stage_bytes);
        uint64_t* bars = (uint64_t*)(tab + NS * ND * kPTABW);
        const uint32_t full0 = afptx::smem_addr(bars), empty0 = full0 + 8 * NS;
        const int cbeg = __ldg(a.chkoff + jb), nchk = __ldg(a.chkoff + jb + 1) - cbeg;

        if (threadIdx.x == 0) {
            for (int s = 0; s < NS; s++) {
                afptx::mbar_init(full0 + 8 * s, 1);
                afptx::mbar_init(empty0 + 8 * s, NW);
            }
            afptx::fence_mbar_init();
        }
        __syncthreads();

        if (warp == NW) {
            // ---------------- producer warp: chunk descriptors two ahead, slot records one ahead
            const int64_t dt = t0 - a.T0;
            int2 cda = load_cd(a, cbeg, nchk, 0), cdb = load_cd(a, cbeg, nchk, 1);
            int2 rcur = make_int2(0, 0), rnxt = make_int2(0, 0);
            int64_t scur = 0, snxt = 0;
            if (lane < cda.x) {
                rcur = __ldg(a.srec + cda.y + lane);
                scur = __ldg(a.soff + cda.y + lane) + dt;
            }
            int kk = 0;
            for (; kk < nchk; kk++) {
                const int st = kk % NS;
                const int2 cdc = load_cd(a, cbeg, nchk, kk + 2);
                rnxt = make_int2(0, 0);
                if (lane < cdb.x) {
                    rnxt = __ldg(a.srec + cdb.y + lane);
                    snxt = __ldg(a.soff + cdb.y + lane) + dt;
                }
                if (kk >= NS &&
                    !afptx::mbar_wait_warp(empty0 + 8 * st, (uint32_t)(kk / NS - 1) & 1u, kPWait)) {
                    if (lane == 0) atomicExch(a.err, 1);
                    break;
                }
                produce(a, smem, tab, full0 + 8 * st, cbeg + kk, cda, (uint32_t)rcur.x, (uint32_t)rcur.y, scur, st,
                        lane);
                rcur = rnxt;
                scur = snxt;
                cda = cdb;
                cdb = cdc;
            }
            // (a drain wait that runs out raises the error flag like any other)
            for (int k2 = max(0, kk - NS); k2 < kk; k2++)
                if (!afptx::mbar_wait_warp(full0 + 8 * (k2 % NS), (uint32_t)(k2 / NS) & 1u, kPWait) && lane == 0)
                    atomicExch(a.err, 1);
            return;
        }

        // ---------------- consumer warps: DPW DM rows each
        uint32_t A[DPW][2][kPMG];
        Sums sums;
#pragma unroll
        for (int u = 0; u < DPW; u++)
#pragma unroll
            for (int m = 0; m < kPMG; m++) A[u][0][m] = A[u][1][m] = 0u;
        sums.init(tmem, warp);
        int npacc = 0;
        for (int kk = 0; kk < nchk; kk++) {
            const int st = kk % NS;
            if (!afptx::mbar_wait_warp(full0 + 8 * st, (uint32_t)(kk / NS) & 1u, kPWait)) {
                if (lane == 0) atomicExch(a.err, 1);
                return;
            }
            const uint16_t* tb0 = tab + (st * ND + warp * DPW) * kPTABW;
            const uint8_t* base = smem + (size_t)st * a.stage_bytes + 4 * lane;
#pragma unroll
            for (int u = 0; u < DPW; u++) {
                const uint16_t* tb = tb0 + u * kPTABW;
                const uint2 h = *reinterpret_cast<const uint2*>(tb);  // starts 0, 1; counts 0, 1
                if (u == 0) {  // the chunk's groups: the same number of rows for every DM
                    const int npc = (int)((h.y & 0xFFFFu) + (h.y >> 16));
                    if (npacc + npc > a.flush) {
#pragma unroll
                        for (int v = 0; v < DPW; v++) sums.fold(A[v], v, lane);
                        npacc = 0;
                    }
                    npacc += npc;
                }
#pragma unroll
                for (int r = 0; r < 2; r++) {
                    const int beg = (int)(r == 0 ? h.x & 0xFFFFu : h.x >> 16);
                    const int n = (int)(r == 0 ? h.y & 0xFFFFu : h.y >> 16);
                    const uint16_t* o = tb + 4 + beg;
                    // the next two rows' offsets one iteration ahead (reads past the
                    // bucket stay inside the table and are never used)
                    uint32_t nx = *reinterpret_cast<const uint32_t*>(o);
                    int i = 0;
                    for (; i + 2 <= n; i += 2) {
                        const uint32_t oo = nx;
                        nx = *reinterpret_cast<const uint32_t*>(o + i + 2);
                        const uint8_t* p1 = base + 4u * (oo & 0xFFFFu);
                        const uint8_t* p2 = base + 4u * (oo >> 16);
                        uint32_t w1[kPMG], w2[kPMG];
#pragma unroll
                        for (int m = 0; m < kPMG; m++) {
                            w1[m] = *reinterpret_cast<const uint32_t*>(p1 + 128 * m);
                            w2[m] = *reinterpret_cast<const uint32_t*>(p2 + 128 * m);
                        }
#pragma unroll
                        for (int m = 0; m < kPMG; m++) A[u][r][m] += w1[m] + w2[m];
                    }
                    if (i < n) {
                        const uint8_t* p1 = base + 4u * (nx & 0xFFFFu);
#pragma unroll
                        for (int m = 0; m < kPMG; m++) A[u][r][m] += *reinterpret_cast<const uint32_t*>(p1 + 128 * m);
                    }
                }
            }
            __syncwarp();
            if (lane == 0) afptx::mbar_arrive(empty0 + 8 * st);
        }

        // ---- outputs and fused row sums
#pragma unroll
        for (int u = 0; u < DPW; u++) {
            sums.fold(A[u], u, lane);
            const int orow = __ldg(a.perm + (int)jb * ND + warp * DPW + u);
            long long ssum = 0, ssq = 0;
#pragma unroll
            for (int h = 0; h < 2; h++) {
                uint32_t w[kPMG];
                sums.get(u, h, w);
#pragma unroll
                for (int i = 0; i < 8; i++) {
#pragma unroll
                    for (int k = 0; k < 2; k++) {
                        const int pos = 2 * (lane + 32 * (8 * h + i)) + k;
                        const int64_t t = t0 + pos;
                        const uint32_t v = w[2 * i + k];
                        if (orow >= 0 && pos < kPTTE && t < a.tend) {
                            a.Y[(int64_t)orow * a.nout + t] = (int32_t)v;
                            ssum += (long long)v;
                            ssq += (long long)v * (long long)v;
                        }
                    }
                }
            }
            if (a.stats) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    ssum += __shfl_xor_sync(0xffffffffu, ssum, o);
                    ssq += __shfl_xor_sync(0xffffffffu, ssq, o);
                }
                if (lane == 0 && orow >= 0) {
                    atomicAdd(reinterpret_cast<unsigned long long*>(&a.stats[orow].sum), (unsigned long long)ssum);
                    atomicAdd(reinterpret_cast<unsigned long long*>(&a.stats[orow].sumsq), (unsigned long long)ssq);
                }
            }
        }
    }
};

// Tensor memory of a block with two DM rows per warp: allocated by the producer
// warp; the address is visible to every thread on return.
__device__ __forceinline__ uint32_t pair_tmem_alloc(uint32_t* slot)
{
    if ((int)threadIdx.x >> 5 == kPNW) {
        afumma::tmem_alloc(afptx::smem_addr(slot), kPTM);
        afumma::tmem_relinquish();
    }
    afumma::fence_before_sync();
    __syncthreads();
    afumma::fence_after_sync();
    return *slot;
}

__device__ __forceinline__ void pair_tmem_free(uint32_t tmem)
{
    afumma::fence_before_sync();
    __syncthreads();  // every warp is done with its sums
    afumma::fence_after_sync();
    if ((int)threadIdx.x >> 5 == kPNW) afumma::tmem_dealloc(tmem, kPTM);
}

// Grid = time tiles of the block x DM blocks, DM blocks fastest (a tile's rows
// stay in L2 while every DM block reads them).
template <int NS, int DPW>
__global__ void __launch_bounds__((kPNW + 1) * 32, 1) k_pair_tile(const PairArgs a)
{
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint32_t tslot;
    const uint32_t tmem = DPW == 2 ? pair_tmem_alloc(&tslot) : 0u;
    PairTile<NS, DPW>::run(a, smem, blockIdx.x % a.nblk, a.T0 + (int64_t)(blockIdx.x / a.nblk) * kPTTE, tmem);
    if (DPW == 2) pair_tmem_free(tmem);
}

// Persistent form over many plans' time blocks (a batch of beams): items
// (job, DM block, tile) in job order, DM blocks fastest, handed out by an
// atomic counter; every job carries its own tables, DM rows per warp and
// ring-stage size (the shared memory is sized for the largest).  The ring
// barriers are invalidated and initialised again between items.
template <int NS>
__global__ void __launch_bounds__((kPNW + 1) * 32, 1)
k_pair_persistent(const PairArgs* __restrict__ jobs, const long long* __restrict__ first, int njobs,
                  long long total, unsigned long long* counter)
{
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ long long item_s;
    __shared__ uint32_t tslot;
    const uint32_t tmem = pair_tmem_alloc(&tslot);
    for (;;) {
        if (threadIdx.x == 0) item_s = (long long)atomicAdd(counter, 1ull);
        __syncthreads();
        const long long item = item_s;
        if (item >= total) break;
        int lo = 0, hi = njobs - 1;  // the job holding the item: first[j] <= item < first[j + 1]
        while (lo < hi) {
            const int mid = (lo + hi + 1) / 2;
            if (__ldg(first + mid) <= item) lo = mid;
            else hi = mid - 1;
        }
        const PairArgs& a = jobs[lo];
        const long long local = item - __ldg(first + lo);
        const unsigned jb = (unsigned)(local % a.nblk);
        const int64_t t0 = a.T0 + (local / a.nblk) * kPTTE;
        if (a.dpw == 2) PairTile<NS, 2>::run(a, smem, jb, t0, tmem);
        else PairTile<NS, 1>::run(a, smem, jb, t0, tmem);
        __syncthreads();  // every warp is done with the ring before its barriers are reset
        if (threadIdx.x == 0) {
            const uint32_t bar0 = afptx::smem_addr(smem + (size_t)NS * a.stage_bytes) +
                                  (uint32_t)(NS * kPNW * a.dpw * kPTABW * 2);
            for (int s = 0; s < 2 * NS; s++) afptx::mbar_inval(bar0 + 8 * s);
        }
    }
    pair_tmem_free(tmem);
}

size_t tables_smem(int ns, int dpw) { return (size_t)ns * kPNW * dpw * kPTABW * 2 + 2 * (size_t)ns * 8; }
int rows_wstride(int maxdr) { return (int)r16(kET + maxdr + 4 + 4 + 48); }
size_t rows_smem(int maxdr, int G) { return (size_t)kET + 48 + (size_t)(G - 1) * rows_wstride(maxdr); }

typedef void (*TileKernel)(const PairArgs);
TileKernel tile_kernel(int ns, int dpw)
{
    if (dpw == 2) return ns == 4 ? k_pair_tile<4, 2> : ns == 3 ? k_pair_tile<3, 2> : k_pair_tile<2, 2>;
    return ns == 4 ? k_pair_tile<4, 1> : ns == 3 ? k_pair_tile<3, 1> : k_pair_tile<2, 1>;
}

size_t pair_budget()
{
    if (const char* b = getenv("AFGB_PAIR_BUDGET_MB")) return (size_t)atoll(b) << 20;
    size_t fr = 0, tot = 0;
    cudaMemGetInfo(&fr, &tot);
    return std::min<size_t>((size_t)48 << 30, tot / 5);
}

// Rates measured on GB300 at 2070 MHz (4096-channel workload, 1001 DMs, 3-deep
// ring).  Stage 2 with its copies (its consumers) left out in a throw-away
// build: 24.8 / 17.0 / 13.2 ms of shared loads (17.3 / 17.0 / 17.2 ms of window
// copies, L2 to shared memory) for groups of 2 / 3 / 4 channels in blocks of 15 DM
// rows; both together 24.8 / 19.2 / 18.8 ms, and in blocks of 30 rows, which copy
// 0.65 / 0.68 / 0.72 of the bytes, 25.0 / 17.2 / 14.3 ms.  The rates below are fitted
// to both stages' times of 70 plans (128 to 4096 channels, 64 to 1495 DMs, 11 k to
// 215 k outputs; the fit's errors are 6 and 7 %).
constexpr double kBlockStart = 4.6e-6;  // a stage-2 block's first copies and its stores, per 15 DM rows
constexpr double kBlockNorm = 6.4;      // how far a block's loads and copies overlap
constexpr double kRowRead = 4.7e12;     // stage 2: rows from HBM, overlapping the blocks (6.2-norm)
inline double load_rate(int G) { return G == 4 ? 37.1e12 : G == 3 ? 37.2e12 : 37.5e12; }
inline double copy_rate(int G) { return G == 4 ? 6.8e12 : G == 3 ? 7.2e12 : 7.7e12; }
// stage 1: a launch, a block of the whole GPU, a row's part of one block (8 KB
// written), and a row of the group that has the most, one after another
constexpr double kRowsLaunch = 5.6e-6, kRowPart = 1.1e-9, kRowSerial = 0.37e-6;
inline double rows_block(int G) { return G == 4 ? 8.1e-9 : G == 3 ? 5.0e-9 : 2.9e-9; }
inline double row_rate(int G) { return G == 4 ? 5.2e12 : G == 3 ? 6.2e12 : 6.5e12; }
// The channel tile kernel: a launch, whole waves of one block per SM, each some
// microseconds and a channel's samples after another.  Fitted, with the kernel whose
// warps build their own tables, to 875 plans (8 to 4096 channels, 2 to 1500 DMs, 300
// to 150,000 outputs; error 5 %).
constexpr double kTileLaunch = 4.0e-6, kTileWave = 4.0e-6, kTileChan = 74.1e-9;
// what two launches cost beyond rows_cost on the smallest plans (on the 875 plans,
// 4 / 6 / 8 us: the slower side by more than 5 % in 28 / 26 / 28)
constexpr double kRowsMargin = 6.0e-6;

}  // namespace

int af_pair_tile_outputs() { return kPTTE; }
int af_pair_ring_depth(int ns) { return ns; }

void af_pairs_free(af_pair_tables* T)
{
    cudaFree(T->d_perm);
    cudaFree(T->d_rdelta);
    cudaFree(T->d_gdr);
    cudaFree(T->d_chunks);
    cudaFree(T->d_chkoff);
    cudaFree(T->d_tabs);
    cudaFree(T->d_srec);
    for (auto& l : T->lay) {
        cudaFree(l.d_pinfo);
        cudaFree(l.d_rinfo);
        cudaFree(l.d_rowoff);
        cudaFree(l.d_soff);
    }
    if (T->ps_owned) cudaFree(T->d_ps);
    for (cudaEvent_t ev : T->tev) cudaEventDestroy(ev);
    *T = af_pair_tables();
}

// Host tables of channel groups of G (2 to 4) channels and dpw DM rows per
// consumer warp (once per plan; no CUDA calls).  Leaves T->ok false when the
// plan is not suited: a block whose group needs more than a stage of rows, a
// delta range beyond the stage-1 window, more than 8 rows per group and 15 DM
// rows, or windows that fit no ring shape.
//
// Group q holds channels G q .. G q + G - 1 (fewer in the last group); a row
// is one tuple of delays relative to the group's first channel,
// (D[d][Gq+i] - D[d][Gq])_{i=1..G-1} (0 for a missing channel), and holds the
// sum over the group's channels at those shifts.  Row g spans the delays
// D[d][Gq] of the DMs with its tuple, from B_g (the smallest, rounded down to
// 16) over span_g samples; the group's range starts at ub_q = min_g B_g.
//
// With tiles and time blocks starting at multiples of 8, a consumer's sample
// offset inside its row window, e = D[d][Gq] - (window start & ~7), does not
// depend on the tile, so every warp's bucketed table of (slot, offset) per
// chunk is computed here once; a window starts (t0 - T0) after its position
// for the time block's first tile.
typedef std::array<int32_t, 3> Key;

static void build_groups(af_plan_t p, int G, int dpw, int NS, int optin, const std::vector<int>& order, af_pair_tables* T)
{
    const int nchan = p->nchan, ndm = p->ndm, NW = kPNW * dpw, K = G - 1;  // NW: DM rows of a block
    const int nblk = (ndm + NW - 1) / NW;
    // plane row of a block's w-th DM, ascending (the last one repeated as padding)
    auto dm_of = [&](int j, int w) { return order[std::min(j * NW + w, ndm - 1)]; };
    const int ng = (nchan + G - 1) / G;
    const int32_t* D = p->delays.data();
    auto key_of = [&](const int32_t* row, int c0) {
        Key k = {0, 0, 0};
        for (int i = 1; i < G; i++)
            if (c0 + i < nchan) k[i - 1] = row[c0 + i] - row[c0];
        return k;
    };
    // rows of a group are stored in lexicographic order of their tuples (stage 1
    // keeps partial sums from one to the next); rlook finds a tuple's row
    std::vector<int32_t> rb(ng + 1, 0), rdelta, rB, rspan, ub(ng);
    std::vector<std::pair<Key, int32_t>> rlook;
    std::vector<int2> gdr((size_t)ng * K);
    std::vector<std::pair<Key, int32_t>> v(ndm);  // (tuple, D[d][Gq])
    struct Row {
        Key key;
        int32_t B, span;
    };
    std::vector<Row> rows;
    int maxdr = 0;
    for (int q = 0; q < ng; q++) {
        const int c0 = G * q;
        for (int d = 0; d < ndm; d++) {
            const int32_t* row = D + (size_t)d * nchan;
            v[d] = std::make_pair(key_of(row, c0), row[c0]);
        }
        std::sort(v.begin(), v.end());
        rows.clear();
        for (int d = 0; d < ndm;) {
            int e = d;
            while (e < ndm && v[e].first == v[d].first) e++;
            const int32_t B = v[d].second & ~15;  // the run is sorted by delay
            rows.push_back(Row{v[d].first, B, v[e - 1].second - B});
            d = e;
        }
        const size_t n0 = rB.size();
        for (const Row& r : rows) {
            rlook.push_back(std::make_pair(r.key, (int32_t)rB.size()));
            for (int i = 0; i < K; i++) rdelta.push_back(r.key[i]);
            rB.push_back(r.B);
            rspan.push_back(r.span);
        }
        rb[q + 1] = (int32_t)rB.size();
        ub[q] = *std::min_element(rB.begin() + n0, rB.end());
        for (int i = 0; i < K; i++) {
            int32_t lo = INT32_MAX, hi = INT32_MIN;
            for (const Row& r : rows) {
                lo = std::min(lo, r.key[i]);
                hi = std::max(hi, r.key[i]);
            }
            gdr[(size_t)q * K + i] = make_int2(lo, hi);
            maxdr = std::max(maxdr, hi - lo);
        }
    }
    // window of the groups' first channels' block spread
    int spread = 0;
    for (int j = 0; j < nblk; j++)
        for (int c = 0; c < nchan; c += G) {
            int32_t hi = INT32_MIN;
            int32_t lo = INT32_MAX;
            for (int w = 0; w < NW; w++) {
                const int32_t v0 = D[(size_t)dm_of(j, w) * nchan + c];
                hi = std::max(hi, v0);
                lo = std::min(lo, v0);
            }
            spread = std::max(spread, hi - lo);
        }
    const int64_t rwe = r8((int64_t)spread + 1031);
    if (spread >= (1 << 20) || maxdr > kMaxDr) return;
    // one stage: up to kPSL windows back to back; the widest window must fit
    // (16 bytes stay free for the static shared memory of the persistent form)
    const int stage_bytes = (int)(((size_t)optin - tables_smem(NS, dpw) - 16) / NS) & ~15;
    if (2 * rwe > stage_bytes) return;
    // chunks of whole groups, at most kPSL windows and stage_bytes each, per block; their tables
    struct Ent {
        int slot[2 * kPNW];
        int e[2 * kPNW];
    };
    std::vector<Ent> ents;
    std::vector<int2> chunks;
    std::vector<int32_t> chkoff(nblk + 1, 0), srow, scpart;
    std::vector<int2> srec;  // per slot: window bytes, offset inside its stage
    std::vector<uint16_t> tabs;
    std::vector<Key> dq(NW), S;
    std::vector<int32_t> d0(NW), sdm;
    int open_slots = 0, open_bytes = 0, first_slot = 0;
    std::vector<int> sbyt;  // slot bytes of the open group
    auto flush = [&]() {
        if (ents.empty()) return;
        const size_t base = tabs.size();
        tabs.resize(base + (size_t)NW * kPTABW, 0);
        for (int w = 0; w < NW; w++) {
            uint16_t* tb = tabs.data() + base + (size_t)w * kPTABW;
            int cnt[2] = {0, 0};
            for (const Ent& en : ents) cnt[en.e[w] & 1]++;
            int pos[2] = {0, (cnt[0] + 1) & ~1};  // bucket starts even: offsets load in pairs
            tb[0] = (uint16_t)pos[0];
            tb[1] = (uint16_t)pos[1];
            tb[2] = (uint16_t)cnt[0];
            tb[3] = (uint16_t)cnt[1];
            for (const Ent& en : ents) {
                const int r = en.e[w] & 1;
                // bytes from the stage's start, a multiple of 4 below 2^18
                tb[4 + pos[r]++] = (uint16_t)((srec[first_slot + en.slot[w]].y + 2 * (en.e[w] - r)) / 4);
            }
        }
        chunks.push_back(make_int2(open_slots, first_slot));
        ents.clear();
        open_slots = 0;
        open_bytes = 0;
    };
    for (int j = 0; j < nblk; j++) {
        for (int q = 0; q < ng; q++) {
            const int c0 = G * q;
            for (int w = 0; w < NW; w++) {
                const int32_t* row = D + (size_t)dm_of(j, w) * nchan;
                d0[w] = row[c0];
                dq[w] = key_of(row, c0);
            }
            S.assign(dq.begin(), dq.end());
            std::sort(S.begin(), S.end());
            S.erase(std::unique(S.begin(), S.end()), S.end());
            if ((int)S.size() > kPSL) return;
            // one window per (block, row): from the smallest delay of the block's DMs on that row
            sdm.assign(S.size(), 0);
            sbyt.assign(S.size(), 0);
            int gbytes = 0;
            for (size_t k = 0; k < S.size(); k++) {
                int32_t lo = INT32_MAX, hi = INT32_MIN;
                for (int w = 0; w < NW; w++)
                    if (dq[w] == S[k]) {
                        lo = std::min(lo, d0[w]);
                        hi = std::max(hi, d0[w]);
                    }
                sdm[k] = lo;
                sbyt[k] = (int)(2 * r8((int64_t)(hi - lo) + 1031));
                gbytes += sbyt[k];
            }
            if (gbytes > stage_bytes) return;
            if (open_slots + (int)S.size() > kPSL || open_bytes + gbytes > stage_bytes) flush();
            if (ents.empty()) first_slot = (int)srec.size();
            for (size_t k = 0; k < S.size(); k++) {
                const int g = std::lower_bound(rlook.begin() + rb[q], rlook.begin() + rb[q + 1],
                                               std::make_pair(S[k], INT32_MIN))->second;
                srec.push_back(make_int2(sbyt[k], open_bytes));
                open_bytes += sbyt[k];
                srow.push_back(g);
                scpart.push_back((sdm[k] & ~7) - rB[g]);
            }
            Ent en;
            for (int w = 0; w < NW; w++) {
                const int k = (int)(std::lower_bound(S.begin(), S.end(), dq[w]) - S.begin());
                en.slot[w] = open_slots + k;
                en.e[w] = d0[w] - (sdm[k] & ~7);
            }
            ents.push_back(en);
            open_slots += (int)S.size();
        }
        flush();
        chkoff[j + 1] = (int32_t)chunks.size();
    }
    // rows copied per group and block: beyond 8 for 15 DM rows the copies alone
    // outweigh the loads they save (the reservation weighs the rest)
    const double rows_per_group = (double)srec.size() / ((double)nblk * ng);
    if (rows_per_group > 8.0 * dpw) return;
    double copy = 0;
    for (const int2& r : srec) copy += r.x;
    T->G = G;
    T->dpw = dpw;
    T->np = ng;
    T->nrows = (int)rB.size();
    T->maxdr = maxdr;
    T->rows_per_pair = rows_per_group;
    T->shape = NS;
    T->stage_bytes = stage_bytes;
    T->copy_per_tile = copy;
    T->nblk = nblk;
    T->ndm_pad = nblk * NW;
    T->spread = spread;
    T->h_rb = std::move(rb);
    T->h_ub = std::move(ub);
    T->h_rB = std::move(rB);
    T->h_rspan = std::move(rspan);
    T->h_srow = std::move(srow);
    T->h_scpart = std::move(scpart);
    T->h_rdelta = std::move(rdelta);
    T->h_gdr = std::move(gdr);
    T->h_chunks = std::move(chunks);
    T->h_chkoff = std::move(chkoff);
    T->h_tabs = std::move(tabs);
    T->h_srec = std::move(srec);
    T->h_perm.assign(T->ndm_pad, -1);
    for (int i = 0; i < ndm; i++) T->h_perm[i] = order[i];
    T->ok = true;
}

// Gives up the host copies of what a set's device tables hold.
static void drop_uploaded(af_pair_tables* T)
{
    auto gone = [](auto& h) { std::remove_reference_t<decltype(h)>().swap(h); };
    gone(T->h_rdelta), gone(T->h_gdr), gone(T->h_chunks), gone(T->h_chkoff), gone(T->h_srec), gone(T->h_perm);
    gone(T->h_tabs);
}

// Device copies of a table set and its layouts' arrays (once, when a
// reservation or a batch first uses the set; the host copies go).
static int upload_groups(af_pair_tables* T)
{
    if (T->d_tabs) {
        drop_uploaded(T);
        return AF_OK;
    }
    cudaError_t e = cudaSuccess;
    auto up = [&](auto** d, auto& h) {
        if (e == cudaSuccess) e = cudaMalloc(d, h.size() * sizeof(h[0]));
        if (e == cudaSuccess) e = cudaMemcpy(*d, h.data(), h.size() * sizeof(h[0]), cudaMemcpyHostToDevice);
    };
    up(&T->d_rdelta, T->h_rdelta);
    up(&T->d_gdr, T->h_gdr);
    up(&T->d_chunks, T->h_chunks);
    up(&T->d_chkoff, T->h_chkoff);
    up(&T->d_srec, T->h_srec);
    up(&T->d_perm, T->h_perm);
    for (auto& l : T->lay)
        if (e != cudaSuccess || (e = cudaMalloc(&l.d_pinfo, (size_t)T->np * sizeof(int4))) != cudaSuccess ||
            (e = cudaMalloc(&l.d_rinfo, (size_t)T->nrows * sizeof(int2))) != cudaSuccess ||
            (e = cudaMalloc(&l.d_rowoff, (size_t)T->nrows * 8)) != cudaSuccess ||
            (e = cudaMalloc(&l.d_soff, T->h_srow.size() * 8)) != cudaSuccess)
            break;
    up(&T->d_tabs, T->h_tabs);
    if (e != cudaSuccess) {  // nothing half done: the set can be tried again
        auto drop = [](auto*& d) {
            cudaFree(d);
            d = nullptr;
        };
        drop(T->d_rdelta), drop(T->d_gdr), drop(T->d_chunks), drop(T->d_chkoff), drop(T->d_srec), drop(T->d_perm);
        drop(T->d_tabs);
        for (auto& l : T->lay) drop(l.d_pinfo), drop(l.d_rinfo), drop(l.d_rowoff), drop(l.d_soff);
        return af_cuda_check(e, "group tables");
    }
    drop_uploaded(T);
    return AF_OK;
}

// Plane rows by ascending DM.
static std::vector<int> dm_order(af_plan_t p)
{
    std::vector<int> order(p->ndm);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return p->dms[x] < p->dms[y]; });
    return order;
}

// The tables of the sets that no reservation uses: the rows' sizes, which the
// cost model reads, stay; the rest (about 20 MB a set on 4096 channels and 1001 DMs,
// for the life of the plan and of every beam of a batch) goes, and is built again
// if a later reservation picks the set.
static void drop_unused(af_plan_t p)
{
    for (af_pair_tables& T : p->alt) {
        drop_uploaded(&T);
        std::vector<int32_t>().swap(T.h_srow);
        std::vector<int32_t>().swap(T.h_scpart);
    }
}

// The tables of set T again, where they were dropped (h_srow is empty then: a set
// has at least one row window).
static int restore_groups(af_plan_t p, af_pair_tables* T)
{
    if (!T->h_srow.empty()) return AF_OK;
    int optin = 0;
    AF_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, p->device));
    build_groups(p, T->G, T->dpw, T->shape, optin, dm_order(p), T);
    return AF_OK;
}

// Groups of 2, 3 and 4 channels in blocks of 15 and of 30 DM rows, all kept until
// a reservation picks one; each set is built by its own host thread.
// (AFGB_PAIR_DPW=1|2 keeps to blocks of 15 or of 30.)
int af_pairs_build(af_plan_t p)
{
    int optin = 0;
    AF_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, p->device));
    const std::vector<int> order = dm_order(p);
    int NS = 3;
    if (const char* e = getenv("AFGB_PAIR_STAGES")) NS = std::min(4, std::max(2, atoi(e)));
    const size_t budget = pair_budget();
    int only = 0;
    if (const char* e = getenv("AFGB_PAIR_DPW")) only = atoi(e);
    std::vector<std::future<void>> jobs;
    const bool threads = (int64_t)p->ndm * p->nchan > 2000;  // a thread takes longer to start than a smaller set
    int k = 0;
    for (int G = 2; G <= (p->nchan >= 8 ? 4 : 2); G++)
        for (int dpw = 1; dpw <= 2; dpw++) {
            if (only == 3 - dpw) continue;
            af_pair_tables* T = k == 0 ? &p->pairs : &p->alt[k - 1];
            k++;
            // (both bits: built here, later, if no thread can be had)
            jobs.push_back(std::async(threads ? std::launch::async | std::launch::deferred : std::launch::deferred,
                                      [=, &order] { build_groups(p, G, dpw, NS, optin, order, T); }));
            T->budget = budget;
        }
    for (auto& j : jobs) j.get();
    return AF_OK;
}

// Row g's length for time blocks of L outputs: the last tile of a block
// starts at most L - TTE + span_g into the row, and its window (at most
// span_g + 1031 samples, rounded to 8) must fit: r16(L + 2 span_g + 32).
static int64_t row_len(const af_pair_tables* T, int g, int64_t L) { return r16(L + 2 * (int64_t)T->h_rspan[g] + 32); }

static int64_t rows_elems(const af_pair_tables* T, int64_t L)
{
    int64_t n = 0;
    for (int g = 0; g < T->nrows; g++) n += row_len(T, g, L);
    return n;
}

// Time block length for nout outputs within the budget (0: the rows do not fit).
static int64_t block_len(const af_pair_tables* T, int64_t nout, size_t max_bytes = SIZE_MAX)
{
    if (!T->ok || nout <= 0) return 0;
    const int64_t tiles = (nout + kPTTE - 1) / kPTTE;
    const int64_t cap = (int64_t)(std::min(T->budget, max_bytes) / 2);
    int64_t lo = kMinTiles, hi = tiles;
    if (rows_elems(T, lo * kPTTE) > cap) return 0;
    if (lo >= hi) return hi * kPTTE;
    while (lo < hi) {  // largest tile count within the budget
        const int64_t mid = (lo + hi + 1) / 2;
        if (rows_elems(T, mid * kPTTE) <= cap) lo = mid;
        else hi = mid - 1;
    }
    return lo * kPTTE;
}

// Layout k (0: af_dedisperse, 1: af_search) of the row buffer for time
// blocks of L outputs; waits for the device first when it replaces a layout
// or the buffer (kernels in flight may read them).  Reservation calls only.
static int pairs_layout(af_plan_t p, int k, int64_t L)
{
    af_pair_tables* T = &p->pairs;
    af_pair_tables::Layout& ly = T->lay[k];
    if (ly.L == L) return AF_OK;
    if (int rc = restore_groups(p, T)) return rc;
    if (int rc = upload_groups(T)) return rc;
    drop_unused(p);
    const int64_t need = rows_elems(T, L);
    if (ly.L || (size_t)need * 2 > T->ps_bytes)
        if (int rc = af_cuda_check(cudaDeviceSynchronize(), "pair layout")) return rc;
    if ((size_t)need * 2 > T->ps_bytes) {
        if (!T->ps_owned) return af_set_error(AF_ENOBUFS, "pairs: the shared row buffer is too small");
        cudaFree(T->d_ps);
        T->d_ps = nullptr;
        T->ps_bytes = 0;
        if (cudaError_t e = cudaMalloc(&T->d_ps, (size_t)need * 2)) {
            cudaGetLastError();  // the failed allocation is reported here, not by the next launch
            T->d_ps = nullptr;
            T->lay[0].L = T->lay[1].L = 0;  // nothing is reserved any more
            return af_cuda_check(e, "group rows");
        }
        T->ps_bytes = (size_t)need * 2;
    }
    std::vector<int64_t> rowoff(T->nrows), soff(T->h_srow.size());
    std::vector<int4> pinfo(T->np);
    std::vector<int2> rinfo(T->nrows);
    int64_t off = 0, maxlen = 0;
    for (int q = 0; q < T->np; q++) {
        const int g0 = T->h_rb[q], g1 = T->h_rb[q + 1];
        int64_t end = 0;
        for (int g = g0; g < g1; g++) {
            const int64_t len = row_len(T, g, L);
            rowoff[g] = off;
            off += len;
            const int start = T->h_rB[g] - T->h_ub[q];
            end = std::max(end, (int64_t)start + len);
            rinfo[g] = make_int2(start, (int)len);
        }
        pinfo[q] = make_int4(g0, g1 - g0, T->h_ub[q], (int)end);
        maxlen = std::max(maxlen, end);
    }
    for (size_t i = 0; i < soff.size(); i++) soff[i] = rowoff[T->h_srow[i]] + T->h_scpart[i];
    ly.L = 0;
    cudaError_t e;
    if ((e = cudaMemcpy(ly.d_rowoff, rowoff.data(), rowoff.size() * 8, cudaMemcpyHostToDevice)) != cudaSuccess ||
        (e = cudaMemcpy(ly.d_soff, soff.data(), soff.size() * 8, cudaMemcpyHostToDevice)) != cudaSuccess ||
        (e = cudaMemcpy(ly.d_pinfo, pinfo.data(), pinfo.size() * sizeof(int4), cudaMemcpyHostToDevice)) !=
            cudaSuccess ||
        (e = cudaMemcpy(ly.d_rinfo, rinfo.data(), rinfo.size() * sizeof(int2), cudaMemcpyHostToDevice)) != cudaSuccess)
        return af_cuda_check(e, "pair layout");
    ly.L = L;
    ly.maxlen = maxlen;
    return AF_OK;
}

// Predicted time (s) of group rows T in time blocks of L outputs on nout
// outputs.  A stage-2 block takes the 6.4-norm of its shared loads' and its window
// copies' times at the rates above (they overlap, not quite), and a launch whole
// waves of one block per SM: blocks of 30 DM rows are faster by up to a quarter
// on many waves and slower where 15 rows fill the last wave better (2128 channels,
// 609 DMs, 22 tiles: 902 blocks of 15 in 0.62 ms, 462 of 30 in 0.75 ms).  Stage 1
// is its blocks and the row pieces they write, or, where they are few, the group
// with the most rows.  Not alone (a batch's beams side by side): its share of the
// GPU's time, without launches, unfilled waves and latencies.
static double rows_cost(af_plan_t p, const af_pair_tables* T, int64_t nout, int64_t L, bool alone = true)
{
    const double nsm = p->num_sms > 0 ? p->num_sms : 152;
    const double loads = 2.0 * kPNW * T->dpw * T->np * 64.0 * kPMG / (load_rate(T->G) / nsm);
    const double copies = T->copy_per_tile / T->nblk / (copy_rate(T->G) / nsm);
    const double block = std::pow(std::pow(loads, kBlockNorm) + std::pow(copies, kBlockNorm), 1.0 / kBlockNorm) + kBlockStart * T->dpw;
    auto waves = [&](int64_t outs) {
        const double w = (double)((outs + kPTTE - 1) / kPTTE) * T->nblk / nsm;
        return alone ? std::ceil(w) : w;
    };
    const int64_t full = nout / L, rest = nout - full * L;
    const double times = (double)full + (rest > 0 ? (double)rest / L : 0.0);
    const double s2 = std::pow(std::pow(block * ((double)full * waves(L) + (rest > 0 ? waves(rest) : 0.0)), 6.2) +
                                   std::pow(times * 2.0 * (double)rows_elems(T, L) / kRowRead, 6.2),
                               1.0 / 6.2);
    double blocks1 = 0;
    int most = 0;
    for (int q = 0; q < T->np; q++) {
        int64_t end = 0;
        for (int g = T->h_rb[q]; g < T->h_rb[q + 1]; g++)
            end = std::max(end, (int64_t)T->h_rB[g] - T->h_ub[q] + row_len(T, g, L));
        blocks1 += (double)((end + kET - 1) / kET);
        most = std::max(most, T->h_rb[q + 1] - T->h_rb[q]);
    }
    const double all = blocks1 * rows_block(T->G) + (double)rows_elems(T, L) / kET * kRowPart;
    const double s1 = alone ? times * (kRowsLaunch + std::cbrt(std::pow(all, 3) + std::pow(most * kRowSerial, 3))) : times * all;
    return s1 + s2;
}

// The same at throughput alone, for blocks of 15 DM rows: bytes moved at a rate.
static double rows_rate_cost(af_plan_t p, const af_pair_tables* T, int64_t nout, int64_t L)
{
    const double tiles = (double)((nout + kPTTE - 1) / kPTTE), blocks = (double)((nout + L - 1) / L);
    const double rate = T->G == 4 ? 31e12 : T->G == 3 ? 37e12 : 40e12;  // loads + copies, blocks of 15 DM rows
    const double s2 = (2.0 * T->ndm_pad * T->np * (double)nout + tiles * T->copy_per_tile) / rate;
    const double s1 = (blocks * 2.0 * (double)rows_elems(T, L) + (double)p->nchan * (double)(nout + p->dmax)) /
                      row_rate(T->G);
    return s1 + s2;
}

// Whether set T in time blocks of L outputs is predicted faster than the channel
// tile kernel, for a plan's calls (alone) and for a batch's beams (not alone; its
// autotuner then measures both).  Of the 875
// plans above this picks the slower side by more than 5 % in 26 (at most 1.19
// times); the two kernels' throughputs alone, as of blocks of 15 DM rows and an
// earlier tile kernel, did so in 213 (2.05 times: few DMs of many channels, or few
// outputs of few channels).  128 channels x 1001 DMs x 5000 outputs: rows 76 us,
// tiles 45; 4096 x 16 x 700: rows 154 us, tiles 314.
static bool rows_beat_tile(af_plan_t p, const af_pair_tables* T, int64_t nout, int64_t L, bool alone)
{
    const double nsm = p->num_sms > 0 ? p->num_sms : 152;
    const int64_t tiles = (nout + af_dedisp_tile_outputs() - 1) / af_dedisp_tile_outputs();
    const double waves = (double)tiles * p->tile.nblk / nsm, wave = kTileWave + kTileChan * p->nchan;
    if (!alone) return rows_cost(p, T, nout, L, false) < waves * wave;
    return rows_cost(p, T, nout, L) + kRowsMargin < kTileLaunch + std::ceil(waves) * wave;
}

// Gives up a table set's row buffer and layouts (after the device is idle).
static int pairs_release(af_pair_tables* T)
{
    if (!T->d_ps && !T->lay[0].L && !T->lay[1].L) return AF_OK;
    if (int rc = af_cuda_check(cudaDeviceSynchronize(), "group rows release")) return rc;
    if (T->ps_owned) cudaFree(T->d_ps);
    T->d_ps = nullptr;
    T->ps_bytes = 0;
    T->ps_owned = true;
    T->lay[0].L = T->lay[1].L = 0;
    return AF_OK;
}

// Picks the group rows for nout outputs: of the group sizes (2 only unless
// larger groups are allowed; AFGB_PAIR_GROUP=2|3|4 restricts), the one
// predicted fastest within max_bytes of rows, if it beats the channel tile
// kernel (AFGB_DEDISP_KERNEL=pairs skips that comparison); it becomes
// p->pairs (a previously picked set gives up its buffer).  *L gets its time
// block; 0 when nothing suits.
// The candidate (0: p->pairs, k: p->alt[k - 1]) and time block the pick would
// take, or -1; changes nothing.
static int pairs_choose(af_plan_t p, int64_t nout, bool allow_larger, size_t max_bytes, int64_t* L, bool alone = true)
{
    *L = 0;
    // the set the model predicts fastest: over 70 plans 0.1 % slower on average than
    // the set that measured fastest, at most 3.2 % (the set of 15-row blocks that moves
    // the fewest bytes, over 47 of them: 6.6 % and 29 %)
    int best = -1;
    double best_t = 0;
    int64_t Ls[6] = {};
    for (int k = 0; k < 6; k++) {
        const af_pair_tables* T = k == 0 ? &p->pairs : &p->alt[k - 1];
        if (!T->ok || (T->G != 2 && !allow_larger) || (p->force_group && T->G != p->force_group)) continue;
        Ls[k] = block_len(T, nout, max_bytes);
        if (Ls[k] <= 0) continue;
        const double t = rows_cost(p, T, nout, Ls[k]);
        if (best < 0 || t < best_t) {
            best = k;
            best_t = t;
        }
    }
    if (best < 0) return -1;
    const bool tile = p->tile.ns1 > 0;  // else the one-thread-per-output kernel
    if (!p->force_pairs && tile && !rows_beat_tile(p, best == 0 ? &p->pairs : &p->alt[best - 1], nout, Ls[best], alone))
        return -1;
    *L = Ls[best];
    return best;
}

int af_pairs_pick(af_plan_t p, int64_t nout, bool allow_larger, size_t max_bytes, int64_t* L, bool alone)
{
    const int best = pairs_choose(p, nout, allow_larger, max_bytes, L, alone);
    if (best < 0) return AF_OK;
    if (best > 0) {
        if (int rc = pairs_release(&p->pairs)) return rc;
        std::swap(p->pairs, p->alt[best - 1]);
    }
    return AF_OK;
}

size_t af_pairs_workspace(af_plan_t p, int64_t nout)
{
    int64_t L = 0;
    const int best = pairs_choose(p, nout, true, SIZE_MAX, &L);
    if (best < 0) return 0;
    return 2 * (size_t)rows_elems(best == 0 ? &p->pairs : &p->alt[best - 1], L);
}

size_t af_pairs_lean_bytes(af_plan_t p, int64_t nout, bool allow_larger, size_t max_bytes)
{
    size_t bytes = 0;
    double best = 0;
    for (int dpw = 1; dpw <= 2 && !bytes; dpw++)  // sets of 30-row blocks only where there is no other
        for (int k = 0; k < 6; k++) {
            const af_pair_tables* T = k == 0 ? &p->pairs : &p->alt[k - 1];
            if (!T->ok || T->dpw != dpw || (T->G != 2 && !allow_larger) || (p->force_group && T->G != p->force_group))
                continue;
            const int64_t L = block_len(T, nout, max_bytes);
            if (L <= 0) continue;
            const double r = rows_rate_cost(p, T, nout, L);
            if (!bytes || r < best) {
                best = r;
                bytes = 2 * (size_t)rows_elems(T, L);
            }
        }
    return bytes;
}

static int reserve_once(af_plan_t p, int64_t nout, int64_t search, bool allow_larger, size_t max_bytes)
{
    int64_t best_L = 0;
    if (int rc = af_pairs_pick(p, nout, allow_larger, max_bytes, &best_L, true)) return rc;
    if (best_L <= 0) return AF_OK;
    af_pair_tables* T = &p->pairs;
    if (best_L > T->lay[0].L)
        if (int rc = pairs_layout(p, 0, best_L)) return rc;
    if (search > 0) {
        // af_search's growing time blocks, so that the input copy overlaps the
        // work: the layout holds the longest of them
        const std::vector<int64_t> blocks = af_search_block_tiles(p, search, T->lay[0].L / kPTTE);
        const int64_t Lmax = *std::max_element(blocks.begin(), blocks.end()) * kPTTE;
        if (int rc = pairs_layout(p, 1, Lmax)) return rc;
    }
    return AF_OK;
}

// Reserves the picked group rows: the row buffer and the layouts of
// af_dedisperse and (with `search`) af_search.  Nothing when none suits.  The set is
// picked, and both layouts are made, for the most outputs any reservation of the plan
// asked for: another length often prefers another set, and a shorter one must not
// give up what a longer one reserved.  Where the device cannot hold the fastest
// set's buffer, the fastest within the lean one where that fits what is free, then
// within half of what is free, a quarter, and so on (shorter time blocks); where not
// even a small block fits, the plan stays on the channel tile kernel.
int af_pairs_reserve(af_plan_t p, int64_t nout, bool search, bool allow_larger, size_t max_bytes)
{
    nout = std::max(nout, p->rows_nout);
    const int64_t srch = std::max(search ? nout : 0, p->rows_search);
    int rc = reserve_once(p, nout, srch, allow_larger, max_bytes);
    if (rc == AF_ENOMEM) {
        size_t fr = 0, tot = 0;
        AF_CUDA(cudaMemGetInfo(&fr, &tot));
        const size_t lean = af_pairs_lean_bytes(p, nout, allow_larger, max_bytes);
        size_t room = std::min(max_bytes, lean && lean <= fr ? lean : fr / 2);
        // ends: no set has a block that fits a small room, and nothing is allocated then
        for (; rc == AF_ENOMEM; room /= 2) rc = reserve_once(p, nout, srch, allow_larger, room);
        if (rc == AF_OK && !af_dedisp_uses_pairs(p, nout) && p->tile.ns1 == 0)
            return af_set_error(AF_ENOMEM, "group rows: no room for a time block's rows");
    }
    if (rc) return rc;
    p->rows_nout = nout;
    p->rows_search = srch;
    return AF_OK;
}

std::vector<int64_t> af_search_block_tiles(af_plan_t p, int64_t nout, int64_t cap_tiles)
{
    // the dedispersion consumes input about 4 times slower than a pinned host copy
    // delivers it, and the copy starts before the first block: each block can be 4
    // times the previous one and still find its input in place when the previous
    // one ends.  262144 samples, 4096 channels, 1001 DMs: a call of 21.9 ms growing
    // by 4 or by 3, 23.4 by 6; 512 channels, 400 DMs, 131072 samples: 1.30 and 1.37
    // ms; 1024 channels, 1001 DMs: 3.64 and 3.60 ms.  A block's tiles are rounded to
    // whole waves of stage-2 blocks, one per SM: without that a block of 18 tiles x
    // 34 DM blocks takes 5 waves for 4.03 of work (that last call: 3.95 ms growing by
    // 6, 3.79 ms with whole waves, before stage 1's present form).
    const int64_t tiles = (nout + kPTTE - 1) / kPTTE;
    const int64_t nsm = p->num_sms > 0 ? p->num_sms : 152, nblk = std::max(1, p->pairs.nblk);
    cap_tiles = std::max<int64_t>(1, cap_tiles);
    auto whole_waves = [&](int64_t t) {
        const int64_t waves = std::max<int64_t>(1, (t * nblk + nsm / 2) / nsm);
        return std::max<int64_t>(1, waves * nsm / nblk);
    };
    std::vector<int64_t> out;
    int64_t b = std::max<int64_t>(1, tiles / 32), done = 0;
    while (done < tiles) {
        const int64_t t = std::min(std::min(whole_waves(b), cap_tiles), tiles - done);
        out.push_back(t);
        done += t;
        b = 4 * t;
    }
    return out;
}

size_t af_pairs_bytes(af_plan_t p, int64_t nout)
{
    const af_pair_tables* T = &p->pairs;
    if (!T->ok || nout <= 0) return 0;
    return 2 * (size_t)rows_elems(T, (nout + kPTTE - 1) / kPTTE * kPTTE);
}

int af_pairs_attach(af_plan_t p, uint16_t* buf, size_t bytes, int64_t nout)
{
    af_pair_tables* T = &p->pairs;
    if (!T->ok) return af_set_error(AF_EINVAL, "pairs: plan cannot use group rows");
    T->lay[0].L = T->lay[1].L = 0;  // until attached: the channel tile kernel
    const int64_t tiles = (nout + kPTTE - 1) / kPTTE;
    const int64_t cap = (int64_t)(bytes / 2);
    int64_t lo = std::min<int64_t>(kMinTiles, tiles), hi = tiles;
    if (rows_elems(T, lo * kPTTE) > cap) return af_set_error(AF_ENOBUFS, "pairs: shared row buffer too small");
    while (lo < hi) {
        const int64_t mid = (lo + hi + 1) / 2;
        if (rows_elems(T, mid * kPTTE) <= cap) lo = mid;
        else hi = mid - 1;
    }
    if (!p->force_pairs && p->tile.ns1 > 0 && !rows_beat_tile(p, T, nout, lo * kPTTE, false))
        return AF_OK;  // this beam stays on the channel tile kernel
    if (int rc = af_cuda_check(cudaDeviceSynchronize(), "pairs attach")) return rc;
    if (T->ps_owned) cudaFree(T->d_ps);
    T->d_ps = buf;
    T->ps_bytes = bytes;
    T->ps_owned = false;
    return pairs_layout(p, 0, lo * kPTTE);
}

int af_launch_pairs_rows(af_plan_t p, const uint8_t* d_in, int64_t nsamp, int layout, int64_t T0, cudaStream_t s,
                         int64_t Lb)
{
    af_pair_tables* T = &p->pairs;
    const af_pair_tables::Layout& ly = T->lay[layout];
    const int64_t L = ly.L;
    if (Lb <= 0) Lb = L;
    if (L <= 0 || L % kPTTE || T0 % kPTTE || Lb > L || Lb % kPTTE)
        return af_set_error(AF_EINVAL, "pairs: time block not laid out");
    const int dshort = (int)((L - Lb) & ~(int64_t)15);
    const size_t s1 = rows_smem(T->maxdr, T->G);
    const void* k1 = T->G == 4   ? (const void*)k_group_rows<4>
                     : T->G == 3 ? (const void*)k_group_rows<3>
                                 : (const void*)k_group_rows<2>;
    if (int rc = af_ensure_smem(k1, s1)) return rc;
    // a block dshort outputs shorter than the layout needs every group's range
    // dshort samples shorter: the grid covers only that
    const int etiles = (int)std::max<int64_t>(1, (ly.maxlen - dshort + kET - 1) / kET);
    const unsigned long long g1 = (unsigned long long)T->np * etiles;
    if (g1 > 0x7fffffffULL) return af_set_error(AF_EINVAL, "pairs: problem too large for one grid");
    if (T->G == 4)
        k_group_rows<4><<<(unsigned)g1, kS1T, s1, s>>>(d_in, nsamp, p->nchan, ly.d_pinfo, T->d_gdr, T->d_rdelta,
                                                      ly.d_rinfo, ly.d_rowoff, T0, etiles, rows_wstride(T->maxdr),
                                                      dshort, T->d_ps);
    else if (T->G == 3)
        k_group_rows<3><<<(unsigned)g1, kS1T, s1, s>>>(d_in, nsamp, p->nchan, ly.d_pinfo, T->d_gdr, T->d_rdelta,
                                                      ly.d_rinfo, ly.d_rowoff, T0, etiles, rows_wstride(T->maxdr),
                                                      dshort, T->d_ps);
    else
        k_group_rows<2><<<(unsigned)g1, kS1T, s1, s>>>(d_in, nsamp, p->nchan, ly.d_pinfo, T->d_gdr, T->d_rdelta,
                                                      ly.d_rinfo, ly.d_rowoff, T0, etiles, rows_wstride(T->maxdr),
                                                      dshort, T->d_ps);
    return af_cuda_check(cudaGetLastError(), "group rows launch");
}

int af_pairs_block_args(af_plan_t p, int64_t nout, int layout, int64_t T0, int32_t* d_plane, af_rowstats_t* d_stats,
                        af_pair_args* out, long long* items, int64_t Lb)
{
    af_pair_tables* T = &p->pairs;
    const af_pair_tables::Layout& ly = T->lay[layout];
    int64_t L = ly.L;
    if (Lb <= 0) Lb = L;
    if (L <= 0 || L % kPTTE || T0 % kPTTE || T0 >= nout || Lb > L || Lb % kPTTE)
        return af_set_error(AF_EINVAL, "pairs: time block not laid out");
    L = Lb;
    af_pair_args& a = *out;
    a.PS = T->d_ps;
    a.chunks = T->d_chunks;
    a.chkoff = T->d_chkoff;
    a.tabs = T->d_tabs;
    a.srec = T->d_srec;
    a.soff = ly.d_soff;
    a.perm = T->d_perm;
    a.stage_bytes = T->stage_bytes;
    a.flush = 65535 / (255 * T->G);
    a.dpw = T->dpw;
    a.nblk = (unsigned)T->nblk;
    a.T0 = T0;
    a.tend = std::min(nout, T0 + L);
    a.nout = nout;
    a.Y = d_plane;
    a.stats = d_stats;
    a.err = p->d_err;
    *items = (long long)((std::min(L, nout - T0) + kPTTE - 1) / kPTTE) * (long long)T->nblk;
    return AF_OK;
}

size_t af_pairs_stage2_smem(af_plan_t p, int ns) { return (size_t)ns * p->pairs.stage_bytes + tables_smem(ns, p->pairs.dpw); }

int af_launch_pairs_persistent(int ns, size_t smem, int grid, const af_pair_args* d_jobs, const long long* d_first,
                               int njobs, long long total, unsigned long long* d_counter, cudaStream_t s)
{
    const auto fn = ns == 4 ? k_pair_persistent<4> : ns == 3 ? k_pair_persistent<3> : k_pair_persistent<2>;
    if (int rc = af_ensure_smem((const void*)fn, smem)) return rc;
    fn<<<grid, (kPNW + 1) * 32, smem, s>>>(d_jobs, d_first, njobs, total, d_counter);
    return af_cuda_check(cudaGetLastError(), "persistent pair tile launch");
}

int af_pairs_ring(af_plan_t p) { return p->pairs.shape; }

int af_launch_pairs_block(af_plan_t p, const uint8_t* d_in, int64_t nsamp, int64_t nout, int32_t* d_plane,
                          af_rowstats_t* d_stats, cudaStream_t s, int layout, int64_t T0, cudaEvent_t* mid, int64_t Lb)
{
    af_pair_tables* T = &p->pairs;
    if (int rc = af_launch_pairs_rows(p, d_in, nsamp, layout, T0, s, Lb)) return rc;
    if (mid) AF_CUDA(cudaEventRecord(*mid, s));
    PairArgs a;
    long long items = 0;
    if (int rc = af_pairs_block_args(p, nout, layout, T0, d_plane, d_stats, &a, &items, Lb)) return rc;
    const size_t s2 = af_pairs_stage2_smem(p, T->shape);
    const TileKernel fn = tile_kernel(T->shape, T->dpw);
    if (int rc = af_ensure_smem((const void*)fn, s2)) return rc;
    if ((unsigned long long)items > 0x7fffffffULL) return af_set_error(AF_EINVAL, "pairs: problem too large for one grid");
    fn<<<(unsigned)items, (kPNW + 1) * 32, s2, s>>>(a);
    return af_cuda_check(cudaGetLastError(), "pair tile launch");
}

int af_launch_pairs(af_plan_t p, const uint8_t* d_in, int64_t nsamp, int64_t nout, int32_t* d_plane,
                    af_rowstats_t* d_stats, cudaStream_t s)
{
    af_pair_tables* T = &p->pairs;
    const int64_t L = T->lay[0].L;
    if (L <= 0) return af_set_error(AF_EINVAL, "pairs: no row buffer reserved");
    if (d_stats)
        if (int rc = af_cuda_check(cudaMemsetAsync(d_stats, 0, (size_t)p->ndm * sizeof(af_rowstats_t), s),
                                   "pairs stats reset"))
            return rc;
    const int slot = T->tcalls > 0 ? T->tnext : -1;
    int b = 0;
    int64_t cut = 0;  // samples by which the last block's rows are shorter
    for (int64_t T0 = 0; T0 < nout; T0 += L, b++) {
        const bool rec = slot >= 0 && b < T->tblocks;
        cudaEvent_t* e = rec ? &T->tev[((size_t)slot * T->tblocks + b) * 3] : nullptr;
        if (rec) AF_CUDA(cudaEventRecord(e[0], s));
        // the last block, or a call shorter than the reservation, needs only its own tiles' rows
        const int64_t Lb = std::min(L, (nout - T0 + kPTTE - 1) / kPTTE * kPTTE);
        cut = (L - Lb) & ~(int64_t)15;
        if (int rc = af_launch_pairs_block(p, d_in, nsamp, nout, d_plane, d_stats, s, 0, T0, rec ? e + 1 : nullptr, Lb))
            return rc;
        if (rec) AF_CUDA(cudaEventRecord(e[2], s));
    }
    if (slot >= 0) {
        T->tnb[slot] = std::min(b, T->tblocks);
        T->trowbytes[slot] = 2 * (rows_elems(T, L) * (int64_t)b - cut * T->nrows);
        T->tcopybytes[slot] = (int64_t)((double)((nout + kPTTE - 1) / kPTTE) * T->copy_per_tile);
        T->tnext = (slot + 1) % T->tcalls;
    }
    return AF_OK;
}

extern "C" int af_dedisperse_timing(af_plan_t p, int ncalls)
try {
    if (int rc = af_check_plan(p)) return rc;
    if (ncalls < 0 || ncalls > 4096) return af_set_error(AF_EINVAL, "af_dedisperse_timing: ncalls in 0..4096");
    af_pair_tables* T = &p->pairs;
    AF_CUDA(cudaDeviceSynchronize());
    for (cudaEvent_t ev : T->tev) cudaEventDestroy(ev);
    T->tev.clear();
    T->tcalls = T->tnext = 0;
    T->tblocks = 8;
    if (ncalls == 0) return AF_OK;
    T->tev.assign((size_t)ncalls * T->tblocks * 3, nullptr);
    for (cudaEvent_t& ev : T->tev)
        if (cudaError_t e = cudaEventCreate(&ev)) return af_cuda_check(e, "af_dedisperse_timing");
    T->tnb.assign(ncalls, 0);
    T->trowbytes.assign(ncalls, 0);
    T->tcopybytes.assign(ncalls, 0);
    T->tcalls = ncalls;
    return AF_OK;
} catch (...) {
    return af_host_exception("af_dedisperse_timing");
}

extern "C" int af_dedisperse_times(af_plan_t p, int call, float* rows_ms, float* tiles_ms, int64_t* row_bytes,
                                   int64_t* copy_bytes)
try {
    if (int rc = af_check_plan(p)) return rc;
    af_pair_tables* T = &p->pairs;
    if (call < 0 || call >= T->tcalls) return af_set_error(AF_EINVAL, "af_dedisperse_times: no such call slot");
    float r = 0.f, t = 0.f;
    for (int b = 0; b < T->tnb[call]; b++) {
        cudaEvent_t* e = &T->tev[((size_t)call * T->tblocks + b) * 3];
        float x = 0.f, y = 0.f;
        AF_CUDA(cudaEventSynchronize(e[2]));
        AF_CUDA(cudaEventElapsedTime(&x, e[0], e[1]));
        AF_CUDA(cudaEventElapsedTime(&y, e[1], e[2]));
        r += x;
        t += y;
    }
    if (rows_ms) *rows_ms = r;
    if (tiles_ms) *tiles_ms = t;
    if (row_bytes) *row_bytes = T->trowbytes[call];
    if (copy_bytes) *copy_bytes = T->tcopybytes[call];
    return AF_OK;
} catch (...) {
    return af_host_exception("af_dedisperse_times");
}
