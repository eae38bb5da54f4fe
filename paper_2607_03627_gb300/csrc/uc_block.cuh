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
// half 4.75 / 5.55 / 7.7 us; with tagged elements 3.4 / 4.1 / 5.1 us.  What is left
// is the chain of one iteration: two stores and tagged loads through L2 (0.5 us
// each), the FP64 instructions of the longest row (up to nine entries, each waiting
// for the one before), and the evaluation.
#pragma once

namespace uc {
namespace dev {

constexpr int kTileRows = 32;          // rows of a tile: one per lane
constexpr int kBlockMaxLps = 64;       // per-LP step data in shared memory
constexpr int kBlockMaxEval = 1024;    // one LP: the weights of a block's iterations in shared memory

// A tile: rows [r0, r0 + rows) of A^T or A; its entries in shared memory as
// columns and values at q * 32 + lane, kmax per lane, beside its vectors.  A long
// column (rows = 1, is_long) spreads its entries over the lanes in the same layout.
struct __align__(16) BlockTile { int r0, rows, lp, aux, kmax, smem, is_long, pad; };
// a warp's tiles: primal ones first
struct BlockWarp { int first, primal, dual, pad; };
struct BlockPlan {
    const BlockTile *tiles;
    const BlockWarp *warps;       // by CTA, then warp
    const unsigned *seq;          // iterations of earlier launches (the evaluation adds this one's)
    ulonglong2 *xt, *yt;          // x-bar and y, tagged
    unsigned long long *stamp;    // kernel timing: the timed iteration's bounds on CTA 0 (or null)
    int stamp_it, nlps, n_eval, head;   // head: bytes before the tiles' part of shared memory
    int pad;
};
struct __align__(16) BlockLp { double tau, nsigma; int j, lim, pad[2]; };

// descriptor, vectors (primal x-bar, x0, c, lower key, upper key; dual y, y0, q),
// values, columns, entries per lane
__host__ __device__ constexpr int tile_bytes(int kmax, bool primal) {
    return (int)sizeof(BlockTile) + kTileRows * (kmax * 12 + (primal ? 40 : 24) + 4);
}

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

// acc + (this lane's entries) . g, in order, N gathers in flight.  g: plain vector
// (the block's start), or tagged and awaited.  Every wait ends: after four seconds
// *stalled is set and the caller leaves.
constexpr unsigned long long kBlockWaitNs = 4000000000ull;
template <int N, bool TAGGED>
__device__ __forceinline__ double tile_dot(double acc, const double *g, const ulonglong2 *gt, unsigned tag, const int *col,
                                           const double *val, int kmax, int cnt, bool &stalled) {
#pragma unroll 1
    for (int e = 0; e < kmax; e += N) {
        double gv[N];
        if (TAGGED) {
            ulonglong2 w[N];
#pragma unroll
            for (int q = 0; q < N; q++) if (e + q < cnt) w[q] = ld_tagged(gt + col[(e + q) * kTileRows]);
            unsigned long long t0 = 0;
            for (unsigned n = 0;; n++) {
                bool ready = true;
#pragma unroll
                for (int q = 0; q < N; q++)
                    if (e + q < cnt && ((unsigned)(w[q].x >> 32) != tag || (unsigned)(w[q].y >> 32) != tag)) {
                        ready = false;
                        w[q] = ld_tagged(gt + col[(e + q) * kTileRows]);
                    }
                if (__all_sync(0xffffffffu, ready)) break;
                if ((n & 255) == 255) {
                    const unsigned long long t = global_ns();
                    if (t0 == 0) t0 = t;
                    if (__any_sync(0xffffffffu, t - t0 > kBlockWaitNs)) { stalled = true; return acc; }
                }
            }
#pragma unroll
            for (int q = 0; q < N; q++) gv[q] = __hiloint2double((int)(unsigned)w[q].y, (int)(unsigned)w[q].x);
        } else {
#pragma unroll
            for (int q = 0; q < N; q++) if (e + q < cnt) gv[q] = g[col[(e + q) * kTileRows]];
        }
#pragma unroll
        for (int q = 0; q < N; q++) {
            if (e + q >= kmax) break;
            if (e + q < cnt) acc = fma(val[(e + q) * kTileRows], gv[q], acc);
        }
    }
    return acc;
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

// Shared memory: the LPs' step data, ONE (a session of one LP): the weights
// {w, 1 - w} of iteration it at it + 1, then the CTA's tiles.  A column keeps x-bar
// (its x is w x-bar + (1 - w) x0, the Halpern step, computed when it is needed
// next).  The last iteration of the block (or before the limit) writes what the
// evaluation and the results read.
template <typename VT, int NT, bool ONE>
__global__ void __launch_bounds__(NT, 1) k_block(const __grid_constant__ BlockPlan P, const __grid_constant__ Bufs b) {
    extern __shared__ __align__(16) unsigned char blk_smem[];
    constexpr int N = NT > 256 ? 4 : 8;   // gathers in flight per row: what the registers hold without spills
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
    // the warp's tiles into shared memory
    const BlockWarp wp = P.warps[blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)];
    unsigned char *pool = blk_smem + P.head;
#pragma unroll 1
    for (int t = 0; t < wp.primal + wp.dual; t++) {
        const BlockTile T = P.tiles[wp.first + t];
        const bool primal = t < wp.primal, ok = lane < T.rows;
        if (lane == 0) *reinterpret_cast<BlockTile *>(pool + T.smem) = T;
        double *vec = reinterpret_cast<double *>(pool + T.smem + sizeof(BlockTile));
        double *val = vec + (primal ? 5 : 3) * kTileRows;
        int *col = reinterpret_cast<int *>(val + T.kmax * kTileRows);
        const int r = T.r0 + lane;
        const int *rp = primal ? b.AT_rp : b.A_rp, *ci = primal ? b.AT_ci : b.A_ci;
        const VT *v = static_cast<const VT *>(primal ? b.AT_v : b.A_v);
        int k0 = 0, k1 = 0, ks = 1;
        if (T.is_long) { k0 = rp[T.r0] + lane; k1 = rp[T.r0 + 1]; ks = 32; }
        else if (ok) { k0 = rp[r]; k1 = rp[r + 1]; }
        for (int q = 0; q < T.kmax; q++) {
            const int k = k0 + q * ks;
            col[q * kTileRows + lane] = k < k1 ? ci[k] : 0;
            val[q * kTileRows + lane] = k < k1 ? widen(v[k]) : 0.0;
        }
        col[T.kmax * kTileRows + lane] = k1 > k0 ? (k1 - k0 + ks - 1) / ks : 0;
        if (ok && primal) {
            vec[lane] = b.x[0][r];
            vec[32 + lane] = b.xa[r];
            vec[64 + lane] = b.c[r];
            vec[96 + lane] = __longlong_as_double(b.lkey[r]);
            vec[128 + lane] = __longlong_as_double(b.ukey[r]);
        } else if (ok) {
            vec[lane] = b.y[0][r];
            vec[32 + lane] = b.ya[r];
            vec[64 + lane] = b.q[r];
        }
    }
    __syncthreads();
    const int nit = nit_;
    unsigned char *const tile0 = wp.primal + wp.dual ? pool + P.tiles[wp.first].smem : pool;   // a warp's tiles lie side by side
    const bool stamps = P.stamp && blockIdx.x == 0 && threadIdx.x == 0;
    const unsigned seq = *P.seq;
    bool stalled = false;
#pragma unroll 1
    for (int it = 0; it < nit; it++) {
        const int src = it & 1;
        const unsigned tag = seq + (unsigned)it + 1;
        if (stamps && it == P.stamp_it) P.stamp[0] = global_ns();
        if (stamps && it == P.stamp_it + 1) P.stamp[1] = global_ns();
        unsigned char *here = tile0;
#pragma unroll 1
        for (int t = 0; t < wp.primal + wp.dual; t++) {
            const int4 ta = *reinterpret_cast<const int4 *>(here), tb = *reinterpret_cast<const int4 *>(here + 16);
            const int r = ta.x + lane, kmax = tb.x;
            double *vec = reinterpret_cast<double *>(here + sizeof(BlockTile));
            const bool ok = lane < ta.y, primal = t < wp.primal, lng = tb.z != 0;
            const BlockLp &L = lps[ONE ? 0 : ta.z];
            const bool keep = it == (ONE ? nit : L.lim) - 1;
            here += tile_bytes(kmax, primal);
            const double *val = vec + (primal ? 5 : 3) * kTileRows + lane;
            const int *col = reinterpret_cast<const int *>(val - lane + kmax * kTileRows) + lane;
            const int cnt = col[kmax * kTileRows];
            if (!ONE && it >= L.lim) continue;
            double acc = lng ? 0.0 : neg_bits(ok ? vec[64 + lane] : 0.0);
            if (primal && it == 0) acc = tile_dot<N, false>(acc, b.y[0], nullptr, 0, col, val, kmax, cnt, stalled);
            else acc = tile_dot<N, true>(acc, nullptr, primal ? P.yt : P.xt, primal ? tag - 1 : tag, col, val, kmax, cnt, stalled);
            if (stalled) break;
            if (primal) {
                if (lng) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                    acc = neg_bits(vec[64]) + acc;
                }
                if (ok) {
                    double x = vec[lane];
                    const double x0 = vec[32 + lane];
                    double2 w = make_double2(0.0, 0.0);
                    if (it > 0) {
                        if (ONE) w = wt[it];
                        else block_weights(b, L.j + it - 1, w.x, w.y);
                        x = fma(w.x, x, w.y * x0);
                    }
                    const double xv = clip_keys(fma(L.tau, acc, x), __double_as_longlong(vec[96 + lane]),
                                                __double_as_longlong(vec[128 + lane]));
                    const double xr = fma(2.0, xv, -x);
                    st_tagged(P.xt + r, xr, tag);
                    vec[lane] = xr;
                    if (keep) {
                        block_weights(b, L.j + it, w.x, w.y);
                        b.x[src][r] = x;
                        b.x[src ^ 1][r] = fma(w.x, xr, w.y * x0);
                        b.xret[r] = xv;
                    }
                }
            } else if (ok) {
                const double y = vec[lane];
                double yv = fma(L.nsigma, acc, y);
                if (r >= ta.w) yv = nonneg(yv);
                double2 w;
                if (ONE) w = wt[it + 1];
                else block_weights(b, L.j + it, w.x, w.y);
                const double yn = fma(w.x, fma(2.0, yv, -y), w.y * vec[32 + lane]);
                st_tagged(P.yt + r, yn, tag);
                vec[lane] = yn;
                if (keep) {
                    b.y[src][r] = y;
                    b.y[src ^ 1][r] = yn;
                    b.yret[r] = yv;
                }
            }
        }
        if (stalled) break;
    }
    if (stalled && lane == 0)
        for (int i = 0; i < P.nlps; i++)
            if (b.S[i].status == RUNNING) { b.S[i].status = STALLED; b.status[i] = STALLED; }
}

}  // namespace dev
}  // namespace uc
