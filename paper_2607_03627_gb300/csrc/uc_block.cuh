// Resident block kernel: all n_eval PDHG iterations between two evaluations in
// one cooperative launch, for sessions whose rows, columns and matrix entries fit
// into the SMs' shared memory (Halpern variant; included by uc_device.cu, which
// defines the arithmetic helpers and the buffers).
//
// An iteration of such an LP is bound by latency, not by work: as two launches it
// takes 8 us at 300 buses (4 us a launch: launch, loads of the row, gathers one
// after another), of which the FP64 pipe needs 0.5.  Here a CTA keeps its rows for
// the whole block, entries and vectors in shared memory, and there is no barrier
// between the halves of an iteration (a grid-wide one costs 1.25 us): every element
// of the gathered vectors carries the iteration it belongs to in the words that
// hold it, and a row waits for just the elements it reads.  One buffer per vector is
// enough: x-bar of column j is overwritten only after j has gathered the new y of
// every row that reads it, so after those rows have read the old x-bar, and the
// same holds for y.
//
// Per iteration, evaluation included (30 / 300 / 1,441 buses of 24 periods): two
// launches 8.05 / 8.25 / 9.4 us; this kernel with a grid-wide barrier after each
// half 4.75 / 5.55 / 7.7 us; with tagged elements 3.4 / 4.1 / 4.9 us.  What is left
// there is the chain of one iteration: two stores and tagged loads through L2 (0.5 us
// each), the FP64 instructions of the longest row (up to nine entries, each waiting
// for the one before), and the evaluation.  Larger LPs are bound by the FP64 pipe:
// 948 k rows and columns (3,000 buses of 48 periods) 14.0 us, of which the pipe needs
// 10.2, and 1.9 M (6,049 buses) 26.9 us of which 20.4; row kernels 18.9 and 33.1.
// They fit because a run's entries are kept once and the rows' constants are read
// from L2: 1.9 M take 164 KB per SM and 2.5 M 205 KB (entries per row and constants
// kept: 474 k at most; entries shared by aligned groups of 8 to 32 rows: 215 KB at
// 1.9 M, and eight LPs of 24 and 48 periods with as many rows did not fit).
#pragma once

namespace uc {
namespace dev {

constexpr int kTileRows = 32;          // rows of a tile: one per lane

// Threads of a CTA, and gathers in flight per row: what the registers hold without
// spills, which live at L2's latency here.  Few tiles: up to eight warps.  Else 24
// warps, or 28 where there are more than kBigTiles tiles per warp of the 24 and the
// pipe's load counts rather than a row's latency: 632 k rows and columns (5.6 tiles)
// 10.1 us with 28, 10.35 with 24, 1.9 M 27.1 and 29.2; but 440 k without angles (4.0, rows
// of up to 16 entries) 14.0 and 12.6.  Gathers with 24 warps, 4 / 5 / 6: 7.9 / 7.4 / 8.4
// us at 55 k without angles, 12.7 / 13.1 / 13.2 at 440 k.  32 warps with 2: 26.9 us
// at 1.9 M, as 28 with 3.
constexpr int kSmallThreads = 256, kSmallN = 8;
constexpr int kMidThreads = 768, kMidN = 4;
constexpr int kBigThreads = 896, kBigN = 3;
constexpr int kBigTiles = 5;
constexpr int kBlockMaxLps = 64;       // per-LP step data in shared memory
constexpr int kBlockMaxEval = UC_RESIDENT_MAX_EVAL;   // one LP: the weights of a block's iterations in shared memory

// A tile: rows [r0, r0 + rows) of A^T or A.  In shared memory: the descriptor's
// first 16 bytes, the rows' own vector (primal x-bar, dual y), then the entries as
// values, as columns, and their counts, once per run.  A run is consecutive rows
// whose entry q is (col_q + s, val_q) for the s-th row, in the device layout mostly one
// constraint or variable of one entity over the periods; bit l of runs is set where a
// run begins at lane l.  Entry q of run g is at g stride + q.  A uniform tile's rows all
// have kmax <= kUniform entries; a long column (one row) spreads its entries over the
// lanes, a run each.
enum TileKind : int { TILE_ANY = 0, TILE_LONG = 1, TILE_UNIFORM = 2 };
struct __align__(16) BlockTile {
    int r0;
    unsigned info;   // see tile_info
    int kmax;
    unsigned runs;
    int smem, img;           // where it is: byte in shared memory, 16-byte unit of the image
    int bytes, pad;          // in shared memory
};
constexpr int kTileHead = 16, kTileOwn = kTileHead + kTileRows * 8;   // before the entries
__host__ __device__ constexpr unsigned tile_info(int rows, int kind, bool primal, bool ineq, int lp) {
    return (unsigned)rows | (unsigned)kind << 6 | (unsigned)primal << 8 | (unsigned)ineq << 9 | (unsigned)lp << 10;
}
__host__ __device__ constexpr int tile_rows(unsigned info) { return info & 63; }
__host__ __device__ constexpr int tile_kind(unsigned info) { return info >> 6 & 3; }
__host__ __device__ constexpr bool tile_primal(unsigned info) { return info >> 8 & 1; }
__host__ __device__ constexpr bool tile_ineq(unsigned info) { return info >> 9 & 1; }
__host__ __device__ constexpr int tile_lp(unsigned info) { return info >> 10; }
// odd where many lanes read a run of their own: no bank is hit twice
__host__ __device__ constexpr int tile_stride(int kmax, int runs) { return runs > 8 ? kmax | 1 : kmax; }
__host__ __device__ constexpr int tile_bytes(int stride, int runs) {
    return kTileOwn + (runs * (stride * 12 + 4) + 15) / 16 * 16;
}
constexpr int kUniform = 4;
// a warp's tiles: primal ones first
struct BlockWarp { int first, count; };
struct BlockPlan {
    const BlockTile *tiles;
    const BlockWarp *warps;       // by CTA, then warp
    unsigned char *image;         // the tiles' entries as they lie in shared memory (k_block_pack)
    const unsigned *seq;          // iterations of earlier launches (the evaluation adds this one's)
    ulonglong2 *xt, *yt;          // x-bar and y, tagged
    unsigned long long *stamp;    // kernel timing: the timed iteration's bounds on CTA 0 (or null)
    int stamp_it, nlps, n_eval, head;   // head: bytes before the warps' staged constants and the tiles
    unsigned polls;               // a wait's limit (LIMIT instance)
};
struct __align__(16) BlockLp { double tau, nsigma; int j, lim, pad[2]; };

constexpr int kStageBytes = 4 * kTileRows * 8;   // a tile's constants: primal c, x0 and the bounds' keys, dual q and y0

// A tagged element: two 64-bit words, each half of the double's bits below the
// tag.  A 64-bit access is never torn, so a word with the right tag has the right
// half, and no fence is needed between data and flag.
__device__ __forceinline__ void st_tagged(ulonglong2 *p, double v, unsigned tag) {
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};"
                 ::"l"(p), "l"(t | (unsigned)__double2loint(v)), "l"(t | (unsigned)__double2hiint(v)) : "memory");
}
__device__ __forceinline__ ulonglong2 ld_tagged(const ulonglong2 *p) {
    ulonglong2 w;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w.x), "=l"(w.y) : "l"(p) : "memory");
    return w;
}

// Every wait ends: after kBlockPolls polls (0.3 to 1 us each) stalled is set and the
// caller leaves.  The CTAs of a cooperative launch start together, once all of them fit
// beside what other streams run (40 SMs held for 20 ms: all 152 CTAs start within 1 us
// of one another after that; two such launches of one CTA per SM run one after the
// other, whatever their streams' priorities), so another kernel delays the launch and
// never an element; the limit, 10 s at least, only ends what a defect would let hang.
// A constant: as a kernel argument 0.6 % of an iteration at 30 to 1,441 buses; the LIMIT
// instance takes it from the plan, for tests of this exit.
constexpr unsigned kBlockPolls = 1u << 25;

// arrived() + (this lane's entries) . g, in order, N gathers in flight; entry q at
// q, its column plus add; g tagged and awaited.  ALL: every lane has N entries.  arrived()
// is called when the first words are there.
template <int N, bool ALL, typename F>
__device__ __forceinline__ double tile_dot(const ulonglong2 *g, unsigned tag, const int *col, const double *val,
                                           int add, int kmax, int cnt, unsigned polls, bool &stalled, F &&arrived) {
    double acc = 0.0;
    g += add;
#pragma unroll 1
    for (int e = 0; e < (ALL ? 1 : kmax); e += N) {
        ulonglong2 w[N];
#pragma unroll
        for (int q = 0; q < N; q++) if (ALL || e + q < cnt) w[q] = ld_tagged(g + col[e + q]);
        for (unsigned n = 0;; n++) {
            bool ready = true;
#pragma unroll
            for (int q = 0; q < N; q++)
                if ((ALL || e + q < cnt) && ((unsigned)(w[q].x >> 32) != tag || (unsigned)(w[q].y >> 32) != tag)) {
                    ready = false;
                    w[q] = ld_tagged(g + col[e + q]);
                }
            if (__all_sync(0xffffffffu, ready)) break;
            if (n > polls) { stalled = true; return acc; }
        }
        if (ALL || e == 0) acc = arrived();
#pragma unroll
        for (int q = 0; q < N; q++) {
            if (!ALL && e + q >= kmax) break;
            if (ALL || e + q < cnt)
                acc = fma(val[e + q], __hiloint2double((int)(unsigned)w[q].y, (int)(unsigned)w[q].x), acc);
        }
    }
    return acc;
}
// the same from a plain vector (the block's start)
__device__ __forceinline__ double plain_dot(double acc, const double *g, const int *col, const double *val, int add, int cnt) {
#pragma unroll 4
    for (int e = 0; e < cnt; e++) acc = fma(val[e], g[col[e] + add], acc);
    return acc;
}

// asynchronous copy of eight bytes to shared memory
__device__ __forceinline__ void copy8(double *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
// of sixteen, past L1
__device__ __forceinline__ void copy16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy8_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ void stage_row(const Bufs &b, double *stage, bool primal, int r) {
    copy8(stage, (primal ? b.c : b.q) + r);
    copy8(stage + 32, (primal ? b.xa : b.ya) + r);
    if (primal) {
        copy8(stage + 64, b.lkey + r);
        copy8(stage + 96, b.ukey + r);
    }
}

__device__ __forceinline__ void block_weights(const Bufs &b, int jj, double &w, double &w1) {
    if (jj < b.nW) {
        w = __ldg(b.W + jj);
        w1 = __ldg(b.W1 + jj);
    } else {
        w = ((double)jj + 1.0) / ((double)jj + 2.0);
        w1 = 1.0 - w;
    }
}

// The image: every tile's entries as k_block's shared memory holds them, made once for
// the tables it belongs to; a warp per tile.
template <typename VT>
__global__ void __launch_bounds__(kSmallThreads) k_block_pack(const BlockTile *__restrict__ tiles, int count, unsigned char *image,
                                                              const __grid_constant__ Bufs b) {
    const int t = blockIdx.x * (kSmallThreads / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (t >= count) return;
    const BlockTile T = tiles[t];
    const bool primal = tile_primal(T.info), lng = tile_kind(T.info) == TILE_LONG;
    const int runs = __popc(T.runs), stride = tile_stride(T.kmax, runs);
    const int at = __popc(T.runs & ((2u << lane) - 1)) - 1;
    double *val = reinterpret_cast<double *>(image + (size_t)T.img * 16);
    int *col = reinterpret_cast<int *>(val + runs * stride);
    if (!(T.runs >> lane & 1)) return;
    const int r = T.r0 + lane;
    const int *rp = primal ? b.AT_rp : b.A_rp, *ci = primal ? b.AT_ci : b.A_ci;
    const VT *v = static_cast<const VT *>(primal ? b.AT_v : b.A_v);
    int k0 = 0, k1 = 0, ks = 1;
    if (lng) { k0 = rp[T.r0] + lane; k1 = rp[T.r0 + 1]; ks = 32; }
    else if (lane < tile_rows(T.info)) { k0 = rp[r]; k1 = rp[r + 1]; }
    for (int q = 0; q < T.kmax; q++) {
        const int k = k0 + q * ks;
        col[at * stride + q] = k < k1 ? ci[k] : 0;
        val[at * stride + q] = k < k1 ? widen(v[k]) : 0.0;
    }
    col[runs * stride + at] = k1 > k0 ? (k1 - k0 + ks - 1) / ks : 0;
}

// Shared memory: the LPs' step data, ONE (a session of one LP): the weights
// {w, 1 - w} of iteration it at it + 1, then the CTA's tiles.  A row's constants come
// from L1 or L2 each iteration, in flight with its gathers: into registers, or in
// the largest CTAs (STAGED), which have none to spare, into kStageBytes of the warp's
// (1.9 M rows and columns 27.1 us; loaded once the gathers are there 29.1).  A column keeps x-bar
// (its x is w x-bar + (1 - w) x0, the Halpern step, computed when it is needed
// next).  The last iteration of the block (or before the limit) writes what the
// evaluation and the results read.
template <typename VT, int NT, bool ONE, bool LIMIT = false>
__global__ void __launch_bounds__(NT, 1) k_block(const __grid_constant__ BlockPlan P, const __grid_constant__ Bufs b) {
    extern __shared__ __align__(16) unsigned char blk_smem[];
    constexpr int N = NT > kMidThreads ? kBigN : NT > kSmallThreads ? kMidN : kSmallN;
    constexpr bool STAGED = NT > kMidThreads;
    __shared__ int nit_;
    BlockLp *lps = reinterpret_cast<BlockLp *>(blk_smem);
    double2 *wt = reinterpret_cast<double2 *>(lps + P.nlps);
    const int lane = threadIdx.x & 31;
    if (threadIdx.x == 0) nit_ = 0;
    __syncthreads();
    int lim = 0;
    for (int i = threadIdx.x; i < P.nlps; i += blockDim.x) {
        const Scalars *S = b.S + i;
        BlockLp L{};
        L.tau = S->tau;
        L.nsigma = -S->sigma;
        L.j = S->j_base;
        L.lim = S->status == RUNNING ? max(0, min(S->n_eval, S->max_iter - S->k_base)) : 0;
        lps[i] = L;
        lim = max(lim, L.lim);
    }
    if (lim > 0) atomicMax(&nit_, lim);
    if (ONE)
        for (int t = threadIdx.x; t <= P.n_eval; t += blockDim.x) {
            double w = 0.0, w1 = 0.0;
            const int jj = b.S->j_base + t - 1;
            if (jj >= 0) block_weights(b, jj, w, w1);
            wt[t] = make_double2(w, w1);
        }
    double *stage = reinterpret_cast<double *>(blk_smem + P.head + (threadIdx.x >> 5) * kStageBytes) + lane;   // STAGED
    // The warp's tiles into shared memory, all copies in flight together: the entries
    // from the image, the vector where it lies (6,049 buses 27.3 us per iteration with
    // the evaluation; row pointers, columns and values one tile after another 27.55).
    const BlockWarp wp = P.warps[blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)];
#pragma unroll 1
    for (int t0 = 0; t0 < wp.count; t0 += 32) {
        BlockTile mine{};
        if (t0 + lane < wp.count) mine = P.tiles[wp.first + t0 + lane];
#pragma unroll 1
        for (int t = 0; t < min(32, wp.count - t0); t++) {
            const int r0 = __shfl_sync(0xffffffffu, mine.r0, t), smem = __shfl_sync(0xffffffffu, mine.smem, t);
            const unsigned info = __shfl_sync(0xffffffffu, mine.info, t);
            const int kmax = __shfl_sync(0xffffffffu, mine.kmax, t), img = __shfl_sync(0xffffffffu, mine.img, t);
            const unsigned starts = __shfl_sync(0xffffffffu, mine.runs, t);
            const int runs = __popc(starts), bytes = tile_bytes(tile_stride(kmax, runs), runs) - kTileOwn;
            unsigned char *here = blk_smem + smem;
            const unsigned char *from = P.image + (size_t)img * 16;
            for (int o = lane * 16; o < bytes; o += 512) copy16(here + kTileOwn + o, from + o);
            if (lane == 0) *reinterpret_cast<int4 *>(here) = make_int4(r0, info, kmax, starts);
            if (lane < tile_rows(info))
                copy8(reinterpret_cast<double *>(here + kTileHead) + lane, (tile_primal(info) ? b.x[0] : b.y[0]) + r0 + lane);
        }
    }
    copy8_wait();
    const unsigned tile0 = wp.count ? P.tiles[wp.first].smem : 0;   // a warp's tiles lie side by side
    __syncthreads();
    const int nit = nit_;
    const bool stamps = P.stamp && blockIdx.x == 0 && threadIdx.x == 0;
    const unsigned seq = *P.seq;
    bool stalled = false;
#pragma unroll 1
    for (int it = 0; it < nit; it++) {
        if (stamps && it == P.stamp_it) P.stamp[0] = global_ns();
        if (stamps && it == P.stamp_it + 1) P.stamp[1] = global_ns();
        unsigned here = tile0;
#pragma unroll 1
        for (int t = 0; t < wp.count; t++) {
            double acc;
            const unsigned tile = here;
            double anchor = 0.0;
            long long lk = 0, uk = 0;
            {
                const int4 T = *reinterpret_cast<const int4 *>(blk_smem + tile);
                const int r = T.x + lane, kmax = T.z, runs = __popc(T.w), stride = tile_stride(kmax, runs);
                const bool ok = lane < tile_rows(T.y), primal = tile_primal(T.y), lng = tile_kind(T.y) == TILE_LONG;
                here += tile_bytes(stride, runs);
                if (!ONE && it >= lps[tile_lp(T.y)].lim) continue;
                // the lane's run and its row in it (lanes without a row: the first)
                const int mine = ok || lng ? lane : 0;
                const unsigned upto = (unsigned)T.w & ((2u << mine) - 1);
                const int at = __popc(upto) - 1, add = mine - (31 - __clz(upto));
                const double *val = reinterpret_cast<const double *>(blk_smem + tile + kTileHead) + kTileRows;
                const int *col = reinterpret_cast<const int *>(val + runs * stride);
                const int cnt = ok || lng ? col[runs * stride + at] : 0;
                val += at * stride;
                col += at * stride;
                // the rows' constants, in flight with the gathers
                double c0 = 0.0;
                if (STAGED) {
                    if (ok) stage_row(b, stage, primal, r);
                } else if (ok) {
                    c0 = __ldg((primal ? b.c : b.q) + r);
                    anchor = __ldg((primal ? b.xa : b.ya) + r);
                    if (NT <= kSmallThreads && primal) { lk = __ldg(b.lkey + r); uk = __ldg(b.ukey + r); }
                }
                auto arrived = [&] {
                    if (STAGED) {
                        copy8_wait();
                        if (ok) c0 = *stage;
                    }
                    return lng ? 0.0 : neg_bits(c0);
                };
                const ulonglong2 *gt = primal ? P.yt : P.xt;
                const unsigned want = seq + (unsigned)it + (primal ? 0u : 1u);
                if (primal && it == 0) {
                    acc = plain_dot(arrived(), b.y[0], col, val, add, cnt);
                } else if (tile_kind(T.y) == TILE_UNIFORM) {
                    if (kmax == 3) acc = tile_dot<3, true>(gt, want, col, val, add, 3, 3, LIMIT ? P.polls : kBlockPolls, stalled, arrived);
                    else if (kmax == 2) acc = tile_dot<2, true>(gt, want, col, val, add, 2, 2, LIMIT ? P.polls : kBlockPolls, stalled, arrived);
                    else if (kmax == 1) acc = tile_dot<1, true>(gt, want, col, val, add, 1, 1, LIMIT ? P.polls : kBlockPolls, stalled, arrived);
                    else acc = tile_dot<4, true>(gt, want, col, val, add, 4, 4, LIMIT ? P.polls : kBlockPolls, stalled, arrived);
                } else acc = tile_dot<N, false>(gt, want, col, val, add, kmax, cnt, LIMIT ? P.polls : kBlockPolls, stalled, arrived);
                if (kmax == 0) acc = arrived();
                if (stalled) break;
                if (lng) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                    acc = neg_bits(__shfl_sync(0xffffffffu, c0, 0)) + acc;
                }
            }
            // the descriptor again: from shared memory, not kept in registers meanwhile
            const int2 d = *reinterpret_cast<const int2 *>(blk_smem + tile);
            const int r = d.x + lane, src = it & 1;
            const unsigned tag = seq + (unsigned)it + 1;
            double *z = reinterpret_cast<double *>(blk_smem + tile + kTileHead) + lane;
            const BlockLp &L = lps[ONE ? 0 : tile_lp(d.y)];
            const bool keep = it == (ONE ? nit : L.lim) - 1;
            if (lane >= tile_rows(d.y)) continue;
            if (STAGED) anchor = stage[32];
            if (tile_primal(d.y)) {
                if (STAGED) {
                    lk = __double_as_longlong(stage[64]);
                    uk = __double_as_longlong(stage[96]);
                } else if (NT > kSmallThreads) {
                    lk = __ldg(b.lkey + r);
                    uk = __ldg(b.ukey + r);
                }
                double x = *z;
                double2 w = make_double2(0.0, 0.0);
                if (it > 0) {
                    if (ONE) w = wt[it];
                    else block_weights(b, L.j + it - 1, w.x, w.y);
                    x = fma(w.x, x, w.y * anchor);
                }
                const double xv = clip_keys(fma(L.tau, acc, x), lk, uk);
                const double xr = fma(2.0, xv, -x);
                st_tagged(P.xt + r, xr, tag);
                *z = xr;
                if (keep) {
                    block_weights(b, L.j + it, w.x, w.y);
                    b.x[src][r] = x;
                    b.x[src ^ 1][r] = fma(w.x, xr, w.y * anchor);
                    b.xret[r] = xv;
                }
            } else {
                const double y = *z;
                double yv = fma(L.nsigma, acc, y);
                if (tile_ineq(d.y)) yv = nonneg(yv);
                double2 w;
                if (ONE) w = wt[it + 1];
                else block_weights(b, L.j + it, w.x, w.y);
                const double yn = fma(w.x, fma(2.0, yv, -y), w.y * anchor);
                st_tagged(P.yt + r, yn, tag);
                *z = yn;
                if (keep) {
                    b.y[src][r] = y;
                    b.y[src ^ 1][r] = yn;
                    b.yret[r] = yv;
                }
            }
        }
        if (stalled) break;
    }
    if (STAGED) copy8_wait();   // a wait that ran out may have left a row's constants in flight
    if (stalled && lane == 0)
        for (int i = 0; i < P.nlps; i++)
            if (b.S[i].status == RUNNING) { b.S[i].status = STALLED; b.status[i] = STALLED; }
}

}  // namespace dev
}  // namespace uc
