// tile.cuh -- the dedispersion tile machinery (Sec. 2.3 brute-force sum),
// templated on the block shape so that the single-plan kernel, the
// persistent multi-beam kernel and the autotuner share one implementation.
//
//   Y[d][t] = sum_c X[c][t + D[d][c]],  0 <= t < nout,  exact int32.
//
// One tile = NW DM rows (one consumer warp each; DMs taken in ascending order
// so a block's delays per channel span the least) x TTE = 128*M - 4 outputs.
// A producer warp streams the channels through shared memory CC = 32 at a
// time in an NS-deep ring (full/empty mbarriers; NS = 4, or 3 / 2 when a
// coarse DM grid widens the windows): for every channel one
// bulk async copy (cp.async.bulk) brings the byte window
// [t0 + Dmin_c, t0 + Dmax_c + 128*M) of that channel, 16-byte aligned, and
// each consumer warp builds its own offset table of the chunk.
//
// Inner loop: lane L of a consumer warp owns outputs t0 + 4*(L + 32*m) + k,
// m < M, k < 4.  For channel c its DM's samples start at byte p = t0 + D; the
// lane reads the ALIGNED 32-bit word at floor4(p) + 4*(L + 32*m) -- one
// conflict-free 128-byte wavefront per warp -- whose bytes are the samples of
// outputs shifted by r = p mod 4.  Channels are therefore bucketed by r and
// each bucket accumulates into its own registers.  The odd bytes are widened
// into 16-bit lanes (at most 256 * 255 per lane between folds), the words
// themselves are summed modulo 2^32, two channels per three-input add:
//     T += w                         (b0 + 2^8 b1 + 2^16 b2 + 2^24 b3)
//     O += prmt(w, 0, 0x4341)        (b1 + 2^16 b3)
// T - 2^8 O is then the sum of b0 + 2^16 b2 modulo 2^32, which is exact
// because both halves stay below 2^16: the even bytes need no masking (4
// integer instructions per two words, against 6).  Every 256 channels (and at
// the end) the buckets are re-aligned as packed 16-bit pairs, one shuffle per
// pair of outputs, and added into output-aligned sums.
//
// Subband mode (SUB = true; stage 1 of the two-stage subband dedispersion,
// Eq. stage1): the rows are coarse DMs, the channels are taken subband after
// subband (cps chunks of 32 per subband, short chunks padded), and at the end
// of every subband the warp folds and stores its partial sums
//     I(j, s, u) = sum_{c in s} X[c][u + D[j][c]]
// as one row of a scratch array.  The table delays are the coarse delays
// minus a per-(row, subband) stagger stag[j][s] = D[j][c_top(s)] - min over
// the block's rows of the same, so the delay spread inside a block is only
// the within-subband dispersion; the warp's output u is then t - stag[j][s].
// Staggers are multiples of 4 outputs, so that a lane's four outputs are one
// aligned 8-byte store (16-bit partial sums, kept packed) or 16-byte store.
// 4096 channels, 126 coarse rows, 64 subbands, 215100 outputs: 6.2 ms, with the
// integer pipe 74 % busy (9.3 ms with one warp building all tables, masked even
// bytes and single 16-bit stores).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"
#include "ptx.cuh"

namespace aftile {

constexpr int CC = 32;                 // channels per stage (one per producer lane)
constexpr int NSTAGE = 4;              // default depth of the shared-memory ring
constexpr int TABW = 40;               // offsets per (stage, warp) table: at most 35 used; the
                                       // slack absorbs one-pair-ahead reads
constexpr uint32_t WAIT_LIMIT = afptx::kMbarWaitPolls;
constexpr int FLUSH_CHUNKS = 256 / CC;

// One beam's dedispersion job (also the argument block of the kernels).
struct TileArgs {
    const uint8_t* X;
    int64_t nsamp;
    int64_t total;          // nchan * nsamp bytes
    int nchan;
    int nchunks;
    const int32_t* dsort;   // [ndm_pad][nchan] delays, DMs ascending
    const int32_t* perm;    // [ndm_pad] output row of each sorted DM, -1 = padding
    const int32_t* dminblk; // [nblk][nchan] smallest delay of each block per channel
    int64_t nout;
    int rw;                 // bytes per channel window (multiple of 16)
    unsigned tiles;
    unsigned nblk;
    int32_t* Y;
    af_rowstats_t* stats;   // may be NULL
    int* err;
    // subband mode only
    int cps;                // chunks per subband
    int nsub;
    const int32_t* sbfirst; // [nsub+1] first channel of each subband
    const int32_t* stag;    // [ndm_pad][nsub] stagger of each row and subband, multiples of 4
    void* I;                // [nrows][nsub][ipitch] uint16 or uint32 partial sums
    int64_t ipitch;         // elements per I row, a multiple of 4
    int64_t li;             // valid outputs per I row in this launch
    int64_t tbase;          // time of tile 0 (the time block's first output)
};

__host__ __device__ constexpr int tte_of(int M) { return 128 * M - 4; }

// Window bytes for a block delay spread (15 bytes alignment slack + spread +
// 128*M bytes read per warp, rounded to 16).
__host__ __device__ inline int window_bytes(int spread, int M) { return (15 + spread + 128 * M + 15) & ~15; }

template <int NW, int NS = NSTAGE>
__host__ __device__ inline size_t smem_bytes(int rw)
{
    return (size_t)NS * CC * rw + (size_t)NS * NW * TABW * sizeof(int) + 2 * NS * 8;
}

__device__ __forceinline__ unsigned lanemask_lt()
{
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// What a tile's sums become: plane rows, or subband partial sums of 16 or 32 bits.
enum Mode { kPlane, kSub16, kSub32 };

template <int NW, int M, Mode MODE = kPlane, int NS = NSTAGE>
struct Tile {
    static constexpr bool SUB = MODE != kPlane;
    // output-aligned sums of one lane and group: two packed pairs, or four words
    static constexpr int NWD = MODE == kSub16 ? 2 : 4;
    static constexpr int NT = (NW + 1) * 32;  // + one producer warp
    static constexpr int TTE = tte_of(M);

    // Walks the chunks: channels [c0, c0 + CC) below cend.  Past the last chunk
    // the range is empty.
    struct Cursor {
        int c0, cend;
        int s, q, next;  // subband mode: subband, chunk within it, its end

        __device__ __forceinline__ void begin(const TileArgs& a)
        {
            if constexpr (SUB) {
                s = q = 0;
                c0 = __ldg(a.sbfirst);
                cend = next = __ldg(a.sbfirst + 1);
            } else {
                c0 = 0;
                cend = a.nchan;
            }
        }
        __device__ __forceinline__ void advance(const TileArgs& a)
        {
            c0 += CC;
            if constexpr (SUB) {
                if (++q == a.cps) {
                    q = 0;
                    s++;
                    c0 = next;
                    cend = next = s < a.nsub ? __ldg(a.sbfirst + s + 1) : next;
                }
            }
        }
    };

    // Producer: the windows of the chunk's channels (lane = channel c, smallest
    // delay dmin in the block) into stage st.  First the tail bytes of windows
    // that end in the last 15 bytes of the input, then the barrier's expected
    // bytes and the bulk copies.
    static __device__ __forceinline__ void produce_chunk(const TileArgs& a, uint8_t* smem, uint32_t full_bar, int c,
                                                         bool valid, int dmin, int st, int64_t t0, int lane)
    {
        int64_t start = 0;
        uint32_t bulk = 0, tail = 0;
        if (valid) {
            start = ((int64_t)c * a.nsamp + t0 + dmin) & ~(int64_t)15;
            int64_t want = min((int64_t)a.rw, a.total - start);
            if constexpr (SUB) want = max((int64_t)0, want);  // staggered tiles may start past the data
            bulk = (uint32_t)(want & ~(int64_t)15);
            tail = (uint32_t)(want - bulk);
        }
        if (valid && tail) {
            uint8_t* sd = smem + (st * CC + lane) * a.rw + bulk;
            for (uint32_t i = 0; i < tail; i++) sd[i] = a.X[start + bulk + i];
        }
        const uint32_t tot = __reduce_add_sync(0xffffffffu, bulk);
        __syncwarp();
        if (lane == 0) {
            afptx::fence_proxy_async();
            afptx::mbar_arrive_expect_tx(full_bar, tot);  // release: tails are visible
        }
        __syncwarp();
        if (valid && bulk) {
            afptx::fence_proxy_async();
            afptx::bulk_g2s(afptx::smem_addr(smem) + (uint32_t)((st * CC + lane) * a.rw), a.X + start, bulk,
                            full_bar);
        }
    }

    // Consumer warp: its row's offsets in the chunk (lane = channel c, delay dl,
    // block's smallest delay dmin), bucketed by r, into tb; beg and cnt are the
    // buckets' first entries and sizes, the same in every lane.  Each warp builds
    // its own table: one warp building all NW was slower than the sums it served.
    static __device__ __forceinline__ void build_table(const TileArgs& a, int* tb, int (&beg)[4], int (&cnt)[4], int c,
                                                       bool valid, int dl, int dmin, int st, int64_t t0, int lane)
    {
        // only the low bits of the channel's address matter
        const uint32_t base = (uint32_t)c * (uint32_t)a.nsamp + (uint32_t)t0;
        const uint32_t r = (base + (uint32_t)dl) & 3u;
        const unsigned v = __ballot_sync(0xffffffffu, valid);
        const unsigned b0 = __ballot_sync(0xffffffffu, r & 1u), b1 = __ballot_sync(0xffffffffu, r & 2u);
        const unsigned mask[4] = {v & ~b0 & ~b1, v & b0 & ~b1, v & ~b0 & b1, v & b0 & b1};
        int s = 0, first = 0;
        unsigned mine = 0;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            beg[k] = s;
            cnt[k] = __popc(mask[k]);
            if (r == k) {
                mine = mask[k];
                first = s;
            }
            s += (cnt[k] + 1) & ~1;  // bucket starts stay even: pairs load as 8 bytes
        }
        if (valid)
            tb[first + __popc(mine & lanemask_lt())] =
                (st * CC + lane) * a.rw + (int)((base + (uint32_t)dmin) & 15u) + (dl - dmin) - (int)r;
    }

    // Adds the four buckets into the output-aligned sums and clears them.  Byte
    // k of bucket r in lane L, group m belongs to output 4*(L + 32*m) + k - r.
    // So output k of lane L takes byte k + r of its own word when k + r <= 3,
    // else byte k + r - 4 of lane L+1's word (lane 0 of group m+1 for L = 31).
    // What a lane owes its left neighbour is added up over the buckets first:
    // outputs (1) and (2, 3) in two packed words, one shuffle each.
    static __device__ __forceinline__ void fold(uint32_t (&T)[4][M], uint32_t (&O)[4][M], uint32_t (&Wd)[M][NWD],
                                                int lane)
    {
        uint32_t c01 = 0u, c23 = 0u;  // group m+1's words, for lane 0
#pragma unroll
        for (int m = M - 1; m >= 0; m--) {
            uint32_t E[4];
#pragma unroll
            for (int r = 0; r < 4; r++) E[r] = T[r][m] - (O[r][m] << 8);
            const uint32_t p01 = E[3] << 16;
            const uint32_t p23 = __byte_perm(E[2], O[2][m], 0x5410) + __byte_perm(O[3][m], E[3], 0x7610) +
                                 (E[1] << 16);
            const int next = (lane + 1) & 31;
            const uint32_t n01 = __shfl_sync(0xffffffffu, lane == 0 ? c01 : p01, next);
            const uint32_t n23 = __shfl_sync(0xffffffffu, lane == 0 ? c23 : p23, next);
            c01 = p01;
            c23 = p23;
            const uint32_t v01 = __byte_perm(E[0], O[0][m], 0x5410) + __byte_perm(O[1][m], E[1], 0x7610) +
                                 __byte_perm(E[2], O[2][m], 0x7632) + (O[3][m] >> 16) + n01;
            const uint32_t v23 = __byte_perm(E[0], O[0][m], 0x7632) + (O[1][m] >> 16) + n23;
            if constexpr (MODE == kSub16) {
                Wd[m][0] += v01;
                Wd[m][1] += v23;
            } else {
                Wd[m][0] += v01 & 0xFFFFu;
                Wd[m][1] += v01 >> 16;
                Wd[m][2] += v23 & 0xFFFFu;
                Wd[m][3] += v23 >> 16;
            }
#pragma unroll
            for (int r = 0; r < 4; r++) T[r][m] = O[r][m] = 0u;
        }
    }

    // Subband mode: writes this warp's sums of subband s as I(row, s, u) with
    // u = t0 - tbase + pos - stag[drow][s], for 0 <= u < li, and clears them.
    // u, TTE and the row pitch are multiples of 4, so four outputs are stored
    // together; up to three past li land in the row's padding.
    static __device__ __forceinline__ void store_subband(const TileArgs& a, int drow, int s, int64_t t0,
                                                         uint32_t (&Wd)[M][NWD], int lane)
    {
        const int orow = __ldg(a.perm + drow);
        if (orow >= 0) {
            const int64_t ub = t0 - a.tbase - (int64_t)__ldg(a.stag + (int64_t)drow * a.nsub + s);
            const int64_t off = ((int64_t)orow * a.nsub + s) * a.ipitch + ub;
            const int lo = (int)max((int64_t)0, min(-ub, (int64_t)TTE));
            const int hi = (int)max((int64_t)0, min(a.li - ub, (int64_t)TTE));
#pragma unroll
            for (int m = 0; m < M; m++) {
                const int pos = 4 * (lane + 32 * m);
                if (pos >= lo && pos < hi) {
                    if constexpr (MODE == kSub16)
                        *reinterpret_cast<uint2*>(reinterpret_cast<uint16_t*>(a.I) + off + pos) =
                            make_uint2(Wd[m][0], Wd[m][1]);
                    else if constexpr (MODE == kSub32)
                        *reinterpret_cast<uint4*>(reinterpret_cast<uint32_t*>(a.I) + off + pos) =
                            make_uint4(Wd[m][0], Wd[m][1], Wd[m][2], Wd[m][3]);
                }
            }
        }
#pragma unroll
        for (int m = 0; m < M; m++)
#pragma unroll
            for (int k = 0; k < NWD; k++) Wd[m][k] = 0u;
    }

    // The whole block computes tile (jb, t0) of job a.  Every thread returns.
    static __device__ __forceinline__ void run(const TileArgs& a, unsigned jb, int64_t t0, uint8_t* smem)
    {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        int* tab = (int*)(smem + (size_t)NS * CC * a.rw);
        uint64_t* bars = (uint64_t*)(tab + NS * NW * TABW);
        const uint32_t full0 = afptx::smem_addr(bars), empty0 = full0 + 8 * NS;

        if (threadIdx.x == 0) {
            for (int s = 0; s < NS; s++) {
                afptx::mbar_init(full0 + 8 * s, 1);
                afptx::mbar_init(empty0 + 8 * s, NW);
            }
            afptx::fence_mbar_init();
        }
        __syncthreads();

        if (warp == NW) {
            // ---------------- producer warp
            // the smallest delays of chunk kk+1 are in flight while chunk kk is produced
            const int32_t* pmin = a.dminblk + (int64_t)jb * a.nchan;
            Cursor cur;
            cur.begin(a);
            int c = cur.c0 + lane;
            bool valid = c < cur.cend;
            int dmin = valid ? __ldg(pmin + c) : 0;
            int kk = 0;
            for (; kk < a.nchunks; kk++) {
                const int st = kk % NS;
                cur.advance(a);
                const int c1 = cur.c0 + lane;
                const bool valid1 = c1 < cur.cend;
                const int dmin1 = valid1 ? __ldg(pmin + c1) : 0;
                if (kk >= NS &&
                    !afptx::mbar_wait_warp(empty0 + 8 * st, (uint32_t)(kk / NS - 1) & 1u, WAIT_LIMIT)) {
                    if (lane == 0) atomicExch(a.err, 1);
                    break;
                }
                produce_chunk(a, smem, full0 + 8 * st, c, valid, dmin, st, t0, lane);
                c = c1;
                valid = valid1;
                dmin = dmin1;
            }
            // leave no copy in flight behind (the consumers normally wait for all of them)
            // (a drain wait that runs out raises the error flag like any other)
            for (int k2 = max(0, kk - NS); k2 < kk; k2++)
                if (!afptx::mbar_wait_warp(full0 + 8 * (k2 % NS), (uint32_t)(k2 / NS) & 1u, WAIT_LIMIT) && lane == 0)
                    atomicExch(a.err, 1);
            return;
        }

        // ---------------- consumer warps: one DM row each
        const int drow = (int)jb * NW + warp;
        uint32_t T[4][M], O[4][M], Wd[M][NWD];
#pragma unroll
        for (int m = 0; m < M; m++) {
#pragma unroll
            for (int r = 0; r < 4; r++) T[r][m] = O[r][m] = 0u;
#pragma unroll
            for (int k = 0; k < NWD; k++) Wd[m][k] = 0u;
        }
        const uint32_t lane4 = (uint32_t)lane * 4u;
        const int32_t* prow = a.dsort + (int64_t)drow * a.nchan;
        const int32_t* pmin = a.dminblk + (int64_t)jb * a.nchan;
        Cursor cur;
        cur.begin(a);
        int c = cur.c0 + lane;
        bool valid = c < cur.cend;
        int dl = valid ? __ldg(prow + c) : 0, dmin = valid ? __ldg(pmin + c) : 0;
        int sb = 0, sq = 0;  // subband mode: current subband and chunk within it
        for (int kk = 0; kk < a.nchunks; kk++) {
            const int st = kk % NS;
            int* tb = tab + (st * NW + warp) * TABW;
            int begs[4], cnts[4];
            build_table(a, tb, begs, cnts, c, valid, dl, dmin, st, t0, lane);
            cur.advance(a);  // the next chunk's delays are in flight meanwhile
            c = cur.c0 + lane;
            valid = c < cur.cend;
            dl = valid ? __ldg(prow + c) : 0;
            dmin = valid ? __ldg(pmin + c) : 0;
            __syncwarp();
            if (!afptx::mbar_wait_warp(full0 + 8 * st, (uint32_t)(kk / NS) & 1u, WAIT_LIMIT)) {
                if (lane == 0) atomicExch(a.err, 1);
                return;
            }
#pragma unroll
            for (int r = 0; r < 4; r++) {
                const int n = cnts[r];
                const int* o = tb + begs[r];
                // the next pair's offsets are loaded one iteration ahead (reads past
                // the bucket stay inside the table and are never used)
                int2 nxt = *reinterpret_cast<const int2*>(o);
                int i = 0;
                for (; i + 2 <= n; i += 2) {
                    const int2 oo = nxt;
                    nxt = *reinterpret_cast<const int2*>(o + i + 2);
                    const uint8_t* p1 = smem + oo.x + lane4;
                    const uint8_t* p2 = smem + oo.y + lane4;
                    uint32_t w1[M], w2[M];
#pragma unroll
                    for (int m = 0; m < M; m++) {
                        w1[m] = *reinterpret_cast<const uint32_t*>(p1 + 128 * m);
                        w2[m] = *reinterpret_cast<const uint32_t*>(p2 + 128 * m);
                    }
#pragma unroll
                    for (int m = 0; m < M; m++) {
                        T[r][m] += w1[m] + w2[m];
                        O[r][m] += __byte_perm(w1[m], 0u, 0x4341) + __byte_perm(w2[m], 0u, 0x4341);
                    }
                }
                if (i < n) {
                    const uint8_t* p1 = smem + nxt.x + lane4;
#pragma unroll
                    for (int m = 0; m < M; m++) {
                        const uint32_t w1 = *reinterpret_cast<const uint32_t*>(p1 + 128 * m);
                        T[r][m] += w1;
                        O[r][m] += __byte_perm(w1, 0u, 0x4341);
                    }
                }
            }
            __syncwarp();
            if (lane == 0) afptx::mbar_arrive(empty0 + 8 * st);  // this warp is done with stage st
            if constexpr (SUB) {
                const bool last = sq == a.cps - 1;
                if ((sq % FLUSH_CHUNKS) == FLUSH_CHUNKS - 1 || last) fold(T, O, Wd, lane);
                if (last) {
                    store_subband(a, drow, sb, t0, Wd, lane);
                    sq = 0;
                    sb++;
                } else {
                    sq++;
                }
            } else {
                if ((kk % FLUSH_CHUNKS) == FLUSH_CHUNKS - 1 || kk == a.nchunks - 1) fold(T, O, Wd, lane);
            }
        }
        if constexpr (!SUB) write_rows(a, drow, t0, Wd, lane);
    }

    // Plane mode: the warp's row of outputs, with its sum and sum of squares.
    static __device__ __forceinline__ void write_rows(const TileArgs& a, int drow, int64_t t0,
                                                      const uint32_t (&Wd)[M][NWD], int lane)
    {
        const int orow = a.perm[drow];
        long long ssum = 0, ssq = 0;
#pragma unroll
        for (int m = 0; m < M; m++) {
            const int pos0 = 4 * (lane + 32 * m);
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const int pos = pos0 + k;
                const int64_t t = t0 + pos;
                const uint32_t v = Wd[m][k];
                if (orow >= 0 && pos < TTE && t < a.nout) {
                    a.Y[(int64_t)orow * a.nout + t] = (int32_t)v;
                    ssum += (long long)v;
                    ssq += (long long)v * (long long)v;
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
};

// Grid = tiles x DM blocks of one job, tile 0 starting at output a.tbase.
// Consecutive blocks take all DM blocks of one time tile, so the input window
// of a time tile stays resident in L2 while every DM block reads it.
template <int NW, int M, int NS = NSTAGE>
__global__ void __launch_bounds__((NW + 1) * 32, 1) k_tile(const TileArgs a)
{
    extern __shared__ __align__(16) uint8_t smem[];
    const unsigned jb = blockIdx.x % a.nblk;
    const int64_t t0 = a.tbase + (int64_t)(blockIdx.x / a.nblk) * Tile<NW, M, kPlane, NS>::TTE;
    Tile<NW, M, kPlane, NS>::run(a, jb, t0, smem);
}

// Stage 1 of the subband dedispersion: grid = tiles x row blocks, tile 0
// starting at a.tbase.
template <int NW, int M, Mode MODE>
__global__ void __launch_bounds__((NW + 1) * 32, 1) k_tile_sb(const TileArgs a)
{
    extern __shared__ __align__(16) uint8_t smem[];
    const unsigned jb = blockIdx.x % a.nblk;
    const int64_t t0 = a.tbase + (int64_t)(blockIdx.x / a.nblk) * Tile<NW, M, MODE>::TTE;
    Tile<NW, M, MODE>::run(a, jb, t0, smem);
}

// Persistent multi-job kernel: each block takes work items (job, DM block,
// time tile) from a global counter until all `total` items are done.  Item i
// belongs to the job b with first[b] <= i < first[b+1]; within a job the
// order is DM block fastest, then time tile.  The job is copied to shared
// memory; the ring's barriers are invalidated and re-initialised per item.
template <int NW, int M>
__global__ void __launch_bounds__((NW + 1) * 32, 1)
k_tile_persistent(const TileArgs* __restrict__ jobs, const long long* __restrict__ first, int njobs,
                  long long total, unsigned long long* counter)
{
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ TileArgs s_job;
    __shared__ long long s_item;
    __shared__ int s_b;
    for (;;) {
        if (threadIdx.x == 0) {
            const long long it = (long long)atomicAdd(counter, 1ull);
            s_item = it;
            int b = 0;
            if (it < total)
                while (b + 1 < njobs && first[b + 1] <= it) b++;
            s_b = b;
            if (it < total) s_job = jobs[b];
        }
        __syncthreads();
        const long long it = s_item;
        if (it >= total) break;
        const long long local = it - first[s_b];
        const unsigned jb = (unsigned)(local % s_job.nblk);
        const int64_t t0 = (int64_t)(local / s_job.nblk) * Tile<NW, M>::TTE;
        Tile<NW, M>::run(s_job, jb, t0, smem);
        __syncthreads();
        if (threadIdx.x == 0) {
            const uint32_t full0 = afptx::smem_addr(smem + (size_t)NSTAGE * CC * s_job.rw +
                                                    (size_t)NSTAGE * NW * TABW * sizeof(int));
            for (int s = 0; s < 2 * NSTAGE; s++) afptx::mbar_inval(full0 + 8 * s);
        }
        __syncthreads();
    }
}

}  // namespace aftile
