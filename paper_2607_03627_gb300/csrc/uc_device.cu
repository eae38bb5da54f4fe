// Device side: restarted, diagonally scaled PDHG for one or several
// (block-diagonally packed) presolved unit-commitment LPs on sm_103a.
//
// The paper's GPU arm solves the LP relaxation with PDHG (Sec. II-C, Alg. 1
// "Solver 1"; Sec. III-C), with an iteration limit of 100,000 and a
// convergence tolerance of 1e-4 (Sec. II-D).  The method is the PDLP scheme
// with a constant step (eta = 0.998 / U, U >= ||A_s||_2 a certified bound, tau = eta / omega,
// sigma = eta * omega):
//
//   x+ = clip(x - tau (c - A^T y), l, u)            k_primal  (A^T row = column of A)
//   y+ = y + sigma (q - A (2 x+ - x)),  y+_I >= 0   k_dual
//   every n_eval iterations: KKT of the current point and of the average
//   since the last restart (k_eval, FP64, deterministic block partials),
//   then the stopping test, restart test and primal-weight update on the
//   device (k_control) and the restart itself (k_apply).
//
// The path is a sparse, bandwidth-bound contraction (about 0.25 flop/byte),
// so no tensor cores are used: every row of A and A^T is owned by one thread,
// vectors are FP64, matrix values FP64 or FP32 (accumulation in FP64).
// n_eval iterations plus the evaluation are captured once in a CUDA graph and
// replayed; the host only polls the LPs' 4-byte statuses in pinned memory per
// replay.  A session keeps the matrices and iterates resident on the device:
// LPs are reset, re-solved, warm-started or replaced (same matrix, new
// right-hand side and bounds) without another upload of the matrix.

#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <atomic>
#include <chrono>
#include <climits>
#include <cmath>
#include <cstring>
#include <functional>
#include <limits>
#include <queue>
#include <thread>
#include <vector>

#include "uc_internal.h"

namespace uc {
namespace dev {

constexpr int kThreads = 256;      // threads per CTA of the row kernels (8 warps)
// Rows handled by one CTA of the evaluation kernel, by the LP's rows + columns
// (not the session's: a batch evaluates each LP as its single solve does).  Small
// LPs take one per thread, so that the evaluation, which the FP64 pipe of the few
// SMs it runs on bounds, spreads over four times the SMs: up to 608 CTAs, four for each
// of 152 SMs, before a CTA gets more.  A constant and not the device's SM count: the sums'
// order, and so the iterates, stay the same on a part of a device.  Evaluation and block
// start at 256 / 512 / 1024 rows: 47 k rows + columns 30.6 / 31.3 / 40.8 us, 157 k 41.0 /
// 42.2 / 43.0, 227 k 48.0 / 46.4 / 50.0, 315 k 56.2 / 53.2 / 53.7, 474 k 76.0 / 68.6 / 63.7.
static int eval_rows(int64_t nm) { return nm <= 256 * 608 ? 256 : nm <= 512 * 608 ? 512 : 1024; }
constexpr int kSlots = 9;          // reduction slots per candidate
constexpr int kPart = 2 * kSlots;  // per-block partial record (current, average)

enum Slot { RP2 = 0, RPU, QY, DY2, RD2, RDU, CX, BND, DX2 };
enum Status { RUNNING = 0, OPTIMAL = 1, ITER_LIMIT = 2, NUMERIC = 3, NEEDS_INIT = 4,
              STALLED = 5,     // a staged kernel gave up waiting for its copies
              INFEASIBLE = 6 };  // a Farkas direction proved the LP primal infeasible
// Halpern variant: every kInfeasEvery-th evaluation tests the dual part of the
// last step's residual, y_hat - y_in, as a primal-infeasibility (Farkas)
// direction; accepted when its objective is positive and its largest
// violation is at most kInfeasEps times that objective (PDLP's test)
constexpr int kInfeasEvery = 4;
constexpr double kInfeasEps = 1e-8;
enum Action { ACT_NONE = 0, ACT_RESTART = 1, ACT_FINISH = 2 };
enum Algo { ALG_HALPERN = 0, ALG_AVERAGE = 1 };
enum Metric { METRIC_KKT = 0, METRIC_FPR = 1, METRIC_FPRP = 2 };

// Per-LP solver state, resident in device memory and only changed by k_control.
struct Scalars {
    double omega, tau, sigma, eta;
    double kkt_anchor, kkt_prev;
    double tol, q_inf, c_inf;
    double rel_p, rel_d, rel_g, abs_p, pobj, dobj;   // of the last evaluated / returned point
    int k_base, j_base, max_iter, n_eval;
    int status, which, action, cand;
    double inv_j;                                    // 1 / iterations averaged at the last evaluation
    int restarts, evals;
    int algo;        // ALG_HALPERN or ALG_AVERAGE
    int metric;      // Halpern restart metric: METRIC_KKT, METRIC_FPR or METRIC_FPRP
    // adaptive step size (averaging variant): trial step, weight of the last
    // attempt (its step if accepted, else 0), step-weighted sum since the
    // restart, buffer of the current iterate, accepted attempts
    int adaptive, ad_src, ad_acc;
    double ad_eta, ad_w, wsum;
    // quotients the kernels would otherwise divide out per thread (an FP64
    // division is a long FP64 sequence): the trial step's tau and sigma, 1 / wsum,
    // and 1 / (steps averaged) at the next evaluation of the constant-step variant
    double ad_tau, ad_sigma, inv_wsum, inv_next;
    // primal-weight controller: gains, running sum and last value of the error
    // e = ln(omega dx / dy) at restarts
    double pw_kp, pw_ki, pw_kd, pw_isum, pw_eprev;
    int pw_has;
    // residual-balance guard on the weight update (0: off, else kappa >= 1)
    double pw_guard;
    // > 0: stop when the largest absolute violation of the unscaled rows is at
    // most this (primal feasibility polishing), instead of the relative KKT test
    double stop_abs;
};
// kkt_anchor / kkt_prev hold the restart metric's anchor and previous value
// for the Halpern variant as well.

// One CTA's slice of rows (or columns) of one LP.
struct Seg {
    int inst;    // LP index
    int begin;   // first global row / column
    int end;     // one past the last
    int aux;     // dual kernel: first ">=" row of this LP; evaluation kernel: 1 for a
                 // column slice, (first ">=" row) << 1 for a row slice
    int rpt;     // iteration kernels: rows per thread (the slice has rpt * blockDim rows)
};

struct Bufs {
    // matrices (block-diagonal when batched, global indices)
    const int *A_rp, *A_ci, *AT_rp, *AT_ci;
    const void *A_v, *AT_v;
    // period-strided 16-row groups: entries per row of group g (or -1) and the
    // group's slot records at 16 g + q (see k_primal)
    const signed char *A_sk, *AT_sk;
    const void *A_sl, *AT_sl;
    // constant vectors
    const double *c, *l, *u, *q, *Dr, *Dc;
    const double *inv_Dr, *inv_Dc;             // 1 / D_r, 1 / D_c (evaluation only)
    const long long *lkey, *ukey;              // order keys of l and u (see okey)
    const double *W, *W1;                      // Halpern weights (j+1)/(j+2) and 1 - that, j < nW
    int nW;
    const double *adS, *adG;                   // adaptive step: 1 - (a+2)^-0.3 and 1 + (a+2)^-0.6, attempt a
    double *adp;                               // adaptive step: per-CTA partial sums of an attempt
    // state: x, y double-buffered
    double *x[2], *y[2];
    double *xsum, *ysum, *xa, *ya, *xret, *yret;   // Halpern: xsum holds x-bar, xret/yret the map output
    unsigned *blk_seq;                         // resident block kernel: iterations of all its launches so far
    int n_eval;
    double *part;                              // per-CTA evaluation records
    double *red;                               // [k][kPart] reduced evaluation records
    Scalars *S;
    int *status;       // [k] copy of each LP's status, read by the host after every replay
};

// ---------------------------------------------------------------------------
// FP64 is scarce on this GPU (2 FMA per SM and clock against 128 in FP32), so
// the kernels spend FP64 instructions only on arithmetic whose rounding
// matters and do selections on the integer pipe, bit-exactly:
//   okey(v)   maps a double to an int64 with the same order (negative values
//             get their magnitude bits flipped); okey is its own inverse, so
//             a bound stored as its key is recovered with okey again;
//   clipping  x to [l, u] compares keys and selects;
//   y_I >= 0  tests the sign bit;
//   FP32 matrix values widen to FP64 by moving exponent and mantissa bits
//             (exact for the normal, nonzero values the presolve guarantees);
//   maxima of non-negative doubles compare their bit patterns.
// ---------------------------------------------------------------------------
__device__ __forceinline__ long long okey(long long b) { return b ^ ((b >> 63) & 0x7fffffffffffffffLL); }

__device__ __forceinline__ double clip_keys(double v, long long lk, long long uk) {
    const long long kv = okey(__double_as_longlong(v));
    if (kv < lk) return __longlong_as_double(okey(lk));
    if (kv > uk) return __longlong_as_double(okey(uk));
    return v;
}

__device__ __forceinline__ double nonneg(double v) {
    return (__double_as_longlong(v) < 0) ? 0.0 : v;
}

__device__ __forceinline__ double widen(double v) { return v; }
// read-once streams (matrix entries, constant vectors, the input iterate) are
// loaded evict-first so that the vector the previous kernel just wrote, which
// this kernel gathers at random, stays in L2.  The row pointers (4 bytes a row)
// are loaded with normal priority and stay in L2 from one iteration to the
// next: they head each row's chain of dependent loads.
template <typename T>
__device__ __forceinline__ T ld_stream(const T *p) { return __ldcs(p); }
__device__ __forceinline__ double widen(float f) {
    const unsigned long long u = __float_as_uint(f);
    const unsigned long long bits = ((u & 0x80000000ull) << 32) | (((u & 0x7fffffffull) << 29) + (896ull << 52));
    return __longlong_as_double((long long)bits);
}

// -v by flipping the sign bit on the integer pipe (exact).  The accumulators of
// the iteration kernels start at -c / -q; written as a plain negation the
// compiler spends an FP64 add on it, one FP64 instruction per row.
__device__ __forceinline__ double neg_bits(double v) {
    int hi = __double2hiint(v);
    asm("xor.b32 %0, %0, 0x80000000;" : "+r"(hi));
    return __hiloint2double(hi, __double2loint(v));
}

// max of two non-negative doubles through their bit patterns
__device__ __forceinline__ double nnmax(double a, double b) {
    return __double_as_longlong(a) >= __double_as_longlong(b) ? a : b;
}

__device__ __forceinline__ void halpern_weights(const Bufs &b, const Scalars *S, int it, double &w, double &w1) {
    const int jj = S->j_base + it;
    if (jj < b.nW) {
        w = b.W[jj];
        w1 = b.W1[jj];
    } else {
        w = ((double)jj + 1.0) / ((double)jj + 2.0);
        w1 = 1.0 - w;
    }
}

// ---------------------------------------------------------------------------
// iteration kernels (one thread per row of A^T or A)
// ---------------------------------------------------------------------------
// Programmatic dependent launch: an iteration kernel launched with the PDL
// attribute may start while its predecessor (the other iteration kernel) is
// still finishing.  Everything it reads before pdl_wait() was written two or
// more launches earlier (every kernel triggers its dependent only after its
// own wait), so only the predecessor's output -- the gathered vector -- is
// read after the wait.  Without the attribute both calls are no-ops.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

constexpr int kPre = 3;   // row entries whose index and value are loaded before the wait

// A session of one LP has uniform tables: CTA c covers rows [c B, c B + B) of
// B = BS * rpt rows, so its slice follows from blockIdx without loading the
// table entry (ntot > 0 marks it; aux = first ">=" row for the dual kernel).
// Rows with more than kLongRow entries (the device layout puts them after all
// others) get a warp each: their slices have rpt = 0 and BS / 32 rows, the
// first cs CTAs covering the n shorter rows.
constexpr int kLongRow = 32;
struct Uniform { int n, aux, rpt, cs, ntot; };
template <int BS>
__device__ __forceinline__ Seg row_slice(const Seg *__restrict__ segs, const Uniform &u) {
    if (u.ntot <= 0) return segs[blockIdx.x];
    if ((int)blockIdx.x < u.cs) {
        const int begin = (int)blockIdx.x * BS * u.rpt;
        return Seg{0, begin, min(begin + BS * u.rpt, u.n), u.aux, u.rpt};
    }
    const int begin = u.n + ((int)blockIdx.x - u.cs) * (BS / 32);
    return Seg{0, begin, min(begin + BS / 32, u.ntot), u.aux, 0};
}

// Period-strided 16-row groups (SD = true).  In the entity-major device layout
// consecutive rows are one constraint (or variable) of one entity in
// consecutive periods.  A group of 16 consecutive rows, g = row / 16, is
// strided when all its rows have k entries and entry q of row s is
// (col_q + s, val_q) for one list of k (col_q, val_q) pairs.  Such a group is
// stored as k slot records at the fixed positions 16 g + q (k <= 16) and
// sk[g] = k; other groups have sk[g] = -1 and keep the CSR path.  A strided
// row thus needs no row pointers and its k slots are read once for 16 rows
// (broadcast to the half-warp, 16x less matrix traffic): its loads are the
// slots and sk[g], all independent of one another, then the gathers of 16
// consecutive elements.  Entry q of a strided row is entry q of its CSR row,
// so the dot product adds the same terms in the same order: iterates are
// identical to the CSR path's, bit for bit.
template <typename VT> struct SlotT;
template <> struct __align__(16) SlotT<double> { int col, pad; double val; };
template <> struct __align__(8) SlotT<float> { int col; float val; };

__device__ __forceinline__ void ld_slot(const SlotT<double> *p, int &col, double &v) {
    const int4 r = __ldg(reinterpret_cast<const int4 *>(p));
    col = r.x;
    v = __hiloint2double(r.w, r.z);
}
__device__ __forceinline__ void ld_slot(const SlotT<float> *p, int &col, double &v) {
    const int2 r = __ldg(reinterpret_cast<const int2 *>(p));
    col = r.x;
    v = widen(__int_as_float(r.y));
}

// The first kPre entries of row r (CSR entries k0 .. k1 - 1, or the group's
// slots): column, value and the row's entry count.  st: the row is in a strided
// group (its slots and sk were loaded before, see the kernels).
template <typename VT, bool SD>
__device__ __forceinline__ int row_head(const int *__restrict__ ci_arr, const VT *__restrict__ v, int k0, int k1,
                                        bool st, int kk, int r, const int (&scol)[kPre], const double (&sval)[kPre],
                                        int (&ci)[kPre], double (&av)[kPre]) {
    if (SD && st) {
#pragma unroll
        for (int q = 0; q < kPre; q++) { ci[q] = scol[q] + (r & 15); av[q] = sval[q]; }
        return kk;
    }
#pragma unroll
    for (int q = 0; q < kPre; q++) {
        ci[q] = 0;
        av[q] = 0.0;
        if (k0 + q < k1) { ci[q] = ld_stream(ci_arr + k0 + q); av[q] = widen(ld_stream(v + k0 + q)); }
    }
    return k1 - k0;
}

// ALGO = ALG_AVERAGE: x+ = clip(x - tau (c - A^T y), l, u), running sum of x+.
// ALGO = ALG_HALPERN: x_hat = that map, x-bar = 2 x_hat - x (gathered by the
// dual kernel), x <- w x-bar + (1 - w) x0 with w = (j+1)/(j+2); x_hat kept at
// the last step of a block (and at the iteration limit).
// 1536 resident threads per SM (40 registers, 12 bytes spilled to L1) for the
// primal kernel and 1280 (48 registers, no spills) for the dual kernel: the
// fastest pair of a sweep over 1024 to 2048 threads.  Both kernels wait on
// memory latency, so more resident rows outweigh the primal kernel's spills.
// The loads of a row are issued before the LP's state is read (the addresses
// are valid either way), so that read overlaps them instead of heading the
// chain of dependent loads.  SD: strided groups read their slots (see above).
// Halpern: an iteration stores x-bar only; its x is the Halpern step from the
// x-bar of the iteration before (it > 0, v) and the anchor x0: 8 bytes per column
// less to store (6,049 buses 33.7 -> 33.1 us per iteration, 2,000 buses with the
// angles eliminated 21.0 -> 19.0; taken before the gathers instead of after them
// it spills and gives 33.5 and 19.5).  The block's last iteration also writes what
// the evaluation and the next block read: x, the next x and the map output.
__device__ __forceinline__ double halpern_x(const Bufs &b, const Scalars *S, int it, int j, double v, double x0) {
    if (it == 0) return v;
    double w, w1;
    halpern_weights(b, S, it - 1, w, w1);
    return fma(w, v, w1 * x0);
}
__device__ __forceinline__ void halpern_store(const Bufs &b, const Scalars *S, int it, int src, int j, double x, double xv, bool keep) {
    const double xb = fma(2.0, xv, -x);
    b.xsum[j] = xb;
    if (!keep) return;
    double w, w1;
    halpern_weights(b, S, it, w, w1);
    b.x[src][j] = x;
    b.x[src ^ 1][j] = fma(w, xb, w1 * b.xa[j]);
    b.xret[j] = xv;
}

// A long column (more than kLongRow entries) gets a warp: the lanes stride over
// its entries, their partial sums are added in a fixed butterfly order, and
// lane 0 adds -c and applies the column's update as the one-thread path does.
template <typename VT, int ALGO>
__device__ __forceinline__ void primal_long(const Seg &sg, const Bufs &b, int it, int src) {
    const int lane = threadIdx.x & 31;
    const int j = sg.begin + (int)(threadIdx.x >> 5);
    if (j >= sg.end) return;                      // whole warps
    const Scalars *S = b.S + sg.inst;
    const VT *__restrict__ v = static_cast<const VT *>(b.AT_v);
    const int k0 = __ldg(b.AT_rp + j), k1 = __ldg(b.AT_rp + j + 1);
    const int k = S->k_base + it;
    if (S->status != RUNNING || k >= S->max_iter) return;
    const bool keep = (it == S->n_eval - 1 || k == S->max_iter - 1);
    pdl_wait();
    pdl_trigger();
    const double *__restrict__ y = b.y[src];
    double part = 0.0;
    for (int e = k0 + lane; e < k1; e += 32) part = fma(widen(ld_stream(v + e)), y[ld_stream(b.AT_ci + e)], part);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if (lane != 0) return;
    const long long lk = ld_stream(b.lkey + j), uk = ld_stream(b.ukey + j);
    const double aux = (ALGO == ALG_AVERAGE) ? b.xsum[j] : ld_stream(b.xa + j);
    const double xin = (ALGO == ALG_AVERAGE) ? ld_stream(b.x[src] + j) : halpern_x(b, S, it, j, it > 0 ? b.xsum[j] : b.x[0][j], aux);
    const double acc = neg_bits(ld_stream(b.c + j)) + part;
    const double xv = clip_keys(fma(S->tau, acc, xin), lk, uk);
    if (ALGO == ALG_AVERAGE) {
        b.x[src ^ 1][j] = xv;
        b.xsum[j] = aux + xv;
    } else {
        halpern_store(b, S, it, src, j, xin, xv, keep);
    }
}

template <typename VT, int ALGO, int BS, bool SD>
__global__ void __launch_bounds__(BS, 1536 / BS) k_primal(const Seg *__restrict__ segs, Bufs b, int it, int src,
                                                           Uniform u) {
    const Seg sg = row_slice<BS>(segs, u);
    if (sg.rpt == 0) {   // a slice of long columns, one per warp
        primal_long<VT, ALGO>(sg, b, it, src);
        return;
    }
    const Scalars *S = b.S + sg.inst;
    const VT *__restrict__ v = static_cast<const VT *>(b.AT_v);
    const SlotT<VT> *__restrict__ slots = static_cast<const SlotT<VT> *>(b.AT_sl);
    const double *__restrict__ y = b.y[src];
    bool waited = false, keep = false;
    for (int t = 0; t < sg.rpt; t++) {
        const int j = sg.begin + t * BS + threadIdx.x;
        if (j >= sg.end) break;
        // independent of the dual kernel that precedes this one
        const int k0 = __ldg(b.AT_rp + j), k1 = __ldg(b.AT_rp + j + 1);
        int kk = -1, scol[kPre];
        double sval[kPre];
        if (SD) {   // the group's k and first slots, whatever path the row takes
            kk = __ldg(b.AT_sk + (j >> 4));
#pragma unroll
            for (int q = 0; q < kPre; q++) ld_slot(slots + (j & ~15) + q, scol[q], sval[q]);
        }
        double xin = (ALGO == ALG_AVERAGE || it == 0) ? ld_stream(b.x[src] + j) : b.xsum[j];
        const long long lk = ld_stream(b.lkey + j), uk = ld_stream(b.ukey + j);
        const double aux = (ALGO == ALG_AVERAGE) ? b.xsum[j] : ld_stream(b.xa + j);
        const bool st = SD && kk >= 0;
        int ci[kPre];
        double av[kPre];
        const int cnt = row_head<VT, SD>(b.AT_ci, v, k0, k1, st, kk, j, scol, sval, ci, av);
        // the accumulator starts at -c, so it ends at A^T y - c
        double acc = neg_bits(ld_stream(b.c + j));
        if (t == 0) {   // the LP's state, read while the row's loads are in flight
            const int k = S->k_base + it;
            if (S->status != RUNNING || k >= S->max_iter) return;
            keep = (it == S->n_eval - 1 || k == S->max_iter - 1);
        }
        if (!waited) { pdl_wait(); pdl_trigger(); waited = true; }
        // a step of the unrolled loop issues only if some lane of the warp needs it
        const unsigned lanes = __activemask();
#pragma unroll
        for (int q = 0; q < kPre; q++) {
            if (!__any_sync(lanes, q < cnt)) break;
            if (q < cnt) acc = fma(av[q], y[ci[q]], acc);
        }
        if (SD && st) {
            for (int q = kPre; q < cnt; q++) {
                int c;
                double a;
                ld_slot(slots + (j & ~15) + q, c, a);
                acc = fma(a, y[c + (j & 15)], acc);
            }
        } else {
            for (int e = k0 + kPre; e < k1; e++) acc = fma(widen(ld_stream(v + e)), y[ld_stream(b.AT_ci + e)], acc);
        }
        if (ALGO == ALG_HALPERN) xin = halpern_x(b, S, it, j, xin, aux);
        const double xv = clip_keys(fma(S->tau, acc, xin), lk, uk);
        if (ALGO == ALG_AVERAGE) {
            b.x[src ^ 1][j] = xv;
            b.xsum[j] = aux + xv;
        } else {
            halpern_store(b, S, it, src, j, xin, xv, keep);
        }
    }
    if (!waited) { pdl_wait(); pdl_trigger(); }
}

// ALGO = ALG_AVERAGE: y+ = proj(y + sigma (q - A (2 x+ - x))), running sum.
// ALGO = ALG_HALPERN: y_hat = proj(y + sigma (q - A x-bar)),
// y <- w (2 y_hat - y) + (1 - w) y0; y_hat kept like x_hat.
template <typename VT, int ALGO, int BS, bool SD>
__global__ void __launch_bounds__(BS, 1536 / BS) k_dual(const Seg *__restrict__ segs, Bufs b, int it, int src,
                                                         Uniform u) {
    const Seg sg = row_slice<BS>(segs, u);
    const Scalars *S = b.S + sg.inst;
    const VT *__restrict__ v = static_cast<const VT *>(b.A_v);
    const SlotT<VT> *__restrict__ slots = static_cast<const SlotT<VT> *>(b.A_sl);
    bool waited = false, keep = false;
    for (int t = 0; t < sg.rpt; t++) {
        const int i = sg.begin + t * BS + threadIdx.x;
        if (i >= sg.end) break;
        const int k0 = __ldg(b.A_rp + i), k1 = __ldg(b.A_rp + i + 1);
        int kk = -1, scol[kPre];
        double sval[kPre];
        if (SD) {
            kk = __ldg(b.A_sk + (i >> 4));
#pragma unroll
            for (int q = 0; q < kPre; q++) ld_slot(slots + (i & ~15) + q, scol[q], sval[q]);
        }
        const double yin = ld_stream(b.y[src] + i);
        const double aux = (ALGO == ALG_AVERAGE) ? b.ysum[i] : ld_stream(b.ya + i);
        const bool st = SD && kk >= 0;
        int ci[kPre];
        double av[kPre];
        const int cnt = row_head<VT, SD>(b.A_ci, v, k0, k1, st, kk, i, scol, sval, ci, av);
        // the accumulator starts at -q, so it ends at A x - q
        double acc = neg_bits(ld_stream(b.q + i));
        if (t == 0) {   // the LP's state, read while the row's loads are in flight
            const int k = S->k_base + it;
            if (S->status != RUNNING || k >= S->max_iter) return;
            keep = (it == S->n_eval - 1 || k == S->max_iter - 1);
        }
        if (!waited) { pdl_wait(); pdl_trigger(); waited = true; }
        const unsigned lanes = __activemask();
        if (ALGO == ALG_AVERAGE) {
            const double *__restrict__ xn = b.x[src ^ 1];
            const double *__restrict__ xo = b.x[src];
#pragma unroll
            for (int q = 0; q < kPre; q++) {
                if (!__any_sync(lanes, q < cnt)) break;
                if (q < cnt) acc = fma(av[q], fma(2.0, xn[ci[q]], -xo[ci[q]]), acc);
            }
            if (SD && st) {
                for (int q = kPre; q < cnt; q++) {
                    int c;
                    double a;
                    ld_slot(slots + (i & ~15) + q, c, a);
                    c += i & 15;
                    acc = fma(a, fma(2.0, xn[c], -xo[c]), acc);
                }
            } else {
                for (int e = k0 + kPre; e < k1; e++) {
                    const int j = b.A_ci[e];
                    acc = fma(widen(v[e]), fma(2.0, xn[j], -xo[j]), acc);
                }
            }
        } else {
            const double *__restrict__ xb = b.xsum;
#pragma unroll
            for (int q = 0; q < kPre; q++) {
                if (!__any_sync(lanes, q < cnt)) break;
                if (q < cnt) acc = fma(av[q], xb[ci[q]], acc);
            }
            if (SD && st) {
                for (int q = kPre; q < cnt; q++) {
                    int c;
                    double a;
                    ld_slot(slots + (i & ~15) + q, c, a);
                    acc = fma(a, xb[c + (i & 15)], acc);
                }
            } else {
                for (int e = k0 + kPre; e < k1; e++) acc = fma(widen(ld_stream(v + e)), xb[ld_stream(b.A_ci + e)], acc);
            }
        }
        double yv = fma(-S->sigma, acc, yin);
        if (i >= sg.aux) yv = nonneg(yv);
        if (ALGO == ALG_AVERAGE) {
            b.y[src ^ 1][i] = yv;
            b.ysum[i] = aux + yv;
        } else {
            double w, w1;
            halpern_weights(b, S, it, w, w1);
            b.y[src ^ 1][i] = fma(w, fma(2.0, yv, -yin), w1 * aux);
            if (keep) b.yret[i] = yv;
        }
    }
    if (!waited) { pdl_wait(); pdl_trigger(); }
}

// ---------------------------------------------------------------------------
// staged iteration kernels (Halpern): persistent CTAs walk a list of row
// chunks; one thread stages each chunk's streamed data -- row pointers,
// column indices and values of its matrix rows and the per-row vectors -- into
// shared memory with bulk asynchronous copies several chunks ahead, so every
// streamed byte is in flight long before it is used and the threads only
// gather the iterate.  Per row the arithmetic is that of k_primal / k_dual,
// operation for operation, so both kernels give identical iterates.
// ---------------------------------------------------------------------------
constexpr int kStRows = 128;     // rows per chunk = threads per CTA
constexpr int kStEnts = 640;     // most matrix entries per chunk
constexpr int kStMaxStages = 8;
constexpr int kStHead = 128;     // bytes before the first stage (the stage barriers)

struct Chunk {
    int inst;    // LP index
    int r0, r1;  // global rows [r0, r1) of A^T (primal) or A (dual)
    int e0, e1;  // their entries [e0, e1)
    int aux;     // dual: first ">=" row of the LP
};

// stage layout: the chunk's descriptor, NV 8-byte vector slices, row
// pointers, column indices, values; every piece is a multiple of 16 bytes, as
// the bulk copies require
template <typename VT, int NV>
struct StLayout {
    static constexpr int kVs = kStRows + 2;                 // doubles per vector slice
    static constexpr int kVec0 = 32;                        // after the descriptor
    static constexpr int kRp = kVec0 + NV * kVs * 8;
    static constexpr int kCi = kRp + (kStRows + 8) * 4;
    static constexpr int kVal = kCi + (kStEnts + 8) * 4;
    static constexpr int kBytes = kVal + (kStEnts + 8) * (int)sizeof(VT);
    static_assert(sizeof(Chunk) <= kVec0 && kRp % 16 == 0 && kCi % 16 == 0 && kVal % 16 == 0 &&
                  kBytes % 16 == 0, "16-byte pieces");
};

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}"
                 ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(smem_addr(bar)), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// wait for a stage, giving up after about a second (the copies are from
// device memory and cannot stall that long unless something is broken)
constexpr unsigned long long kStWaitNs = 1000000000ull;
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity) {
    if (mbar_test(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    for (unsigned n = 1;; n++) {
        if (mbar_test(bar, parity)) return true;
        if ((n & 255) == 0 && global_ns() - t0 > kStWaitNs) return false;
    }
}
__device__ __forceinline__ uint64_t l2_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
// bulk copy of `bytes` (a multiple of 16, both addresses 16-byte aligned) from
// global to this CTA's shared memory, completing on `bar`
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar, uint64_t pol) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
                 ::"r"(smem_addr(dst)), "l"(src), "r"(bytes), "r"(smem_addr(bar)), "l"(pol) : "memory");
}

// the copy window of a chunk: rows and entries rounded out to 16-byte boundaries
template <typename VT>
struct StWindow {
    int r0a, rpa, cia, va;
    uint32_t nv, nrp, nci, nva;   // bytes
    __device__ __forceinline__ StWindow(const Chunk &ch) {
        constexpr int VA = 16 / (int)sizeof(VT);
        r0a = ch.r0 & ~1;
        rpa = ch.r0 & ~3;
        cia = ch.e0 & ~3;
        va = ch.e0 & ~(VA - 1);
        nv = (uint32_t)((ch.r1 - r0a + 1) & ~1) * 8u;
        nrp = (uint32_t)((ch.r1 + 1 - rpa + 3) & ~3) * 4u;
        nci = (uint32_t)((ch.e1 - cia + 3) & ~3) * 4u;
        nva = (uint32_t)((ch.e1 - va + VA - 1) & ~(VA - 1)) * (uint32_t)sizeof(VT);
    }
};

// what an iteration kernel needs of one LP at step `it` of the block: loaded
// when a CTA's chunks move to another LP (each CTA's chunks are grouped by LP)
struct StLp {
    int inst = -1;
    bool live = false, keep = false;
    double step = 0.0, w = 0.0, w1 = 0.0;   // tau (primal) or -sigma (dual); Halpern weights
};
template <bool PRIMAL>
__device__ __forceinline__ void st_load_lp(StLp &L, const Bufs &b, int inst, int it) {
    const Scalars *S = b.S + inst;
    const int k = S->k_base + it;
    L.inst = inst;
    L.live = S->status == RUNNING && k < S->max_iter;
    if (!L.live) return;
    L.keep = (it == S->n_eval - 1 || k == S->max_iter - 1);
    L.step = PRIMAL ? S->tau : -S->sigma;
    halpern_weights(b, S, it, L.w, L.w1);
}

// PRIMAL = true: rows of A^T, vectors x, c, lkey, ukey, x0; gathers y.
// PRIMAL = false: rows of A, vectors y, q, y0; gathers x-bar.
// The descriptor goes into the stage header before the arrive, so the
// threads that wait on the stage barrier see it.
template <typename VT, bool PRIMAL>
__device__ __forceinline__ void st_issue(const Chunk &ch, bool live, unsigned char *sb, uint64_t *bar,
                                         const Bufs &b, int src, uint64_t pol) {
    constexpr int NV = PRIMAL ? 5 : 3;
    using Ly = StLayout<VT, NV>;
    *reinterpret_cast<Chunk *>(sb) = ch;
    if (!live) { mbar_arrive(bar); return; }
    const StWindow<VT> w(ch);
    mbar_expect_tx(bar, NV * w.nv + w.nrp + w.nci + w.nva);
    unsigned char *v = sb + Ly::kVec0;
    constexpr int VB = Ly::kVs * 8;
    if (PRIMAL) {
        bulk_load(v + 0 * VB, b.x[src] + w.r0a, w.nv, bar, pol);
        bulk_load(v + 1 * VB, b.c + w.r0a, w.nv, bar, pol);
        bulk_load(v + 2 * VB, b.lkey + w.r0a, w.nv, bar, pol);
        bulk_load(v + 3 * VB, b.ukey + w.r0a, w.nv, bar, pol);
        bulk_load(v + 4 * VB, b.xa + w.r0a, w.nv, bar, pol);
        bulk_load(sb + Ly::kRp, b.AT_rp + w.rpa, w.nrp, bar, pol);
        if (w.nci) bulk_load(sb + Ly::kCi, b.AT_ci + w.cia, w.nci, bar, pol);
        if (w.nva) bulk_load(sb + Ly::kVal, static_cast<const VT *>(b.AT_v) + w.va, w.nva, bar, pol);
    } else {
        bulk_load(v + 0 * VB, b.y[src] + w.r0a, w.nv, bar, pol);
        bulk_load(v + 1 * VB, b.q + w.r0a, w.nv, bar, pol);
        bulk_load(v + 2 * VB, b.ya + w.r0a, w.nv, bar, pol);
        bulk_load(sb + Ly::kRp, b.A_rp + w.rpa, w.nrp, bar, pol);
        if (w.nci) bulk_load(sb + Ly::kCi, b.A_ci + w.cia, w.nci, bar, pol);
        if (w.nva) bulk_load(sb + Ly::kVal, static_cast<const VT *>(b.A_v) + w.va, w.nva, bar, pol);
    }
}

template <typename VT, bool PRIMAL>
__global__ void __launch_bounds__(kStRows, 8) k_iter_staged(const Chunk *__restrict__ chunks,
                                                            const int *__restrict__ cta_ptr, Bufs b, int it, int src,
                                                            int stages) {
    constexpr int NV = PRIMAL ? 5 : 3;
    using Ly = StLayout<VT, NV>;
    constexpr int VS = Ly::kVs;
    extern __shared__ __align__(128) unsigned char st_smem[];
    uint64_t *bar = reinterpret_cast<uint64_t *>(st_smem);
    unsigned char *stage0 = st_smem + kStHead;
    const int tid = threadIdx.x;
    const int q0 = cta_ptr[blockIdx.x], q1 = cta_ptr[blockIdx.x + 1];
    const uint64_t pol = l2_evict_first();
    if (tid == 0) {
        for (int s = 0; s < stages; s++) mbar_init(bar + s, 1);
        mbar_init_fence();
    }
    __syncthreads();
    // producer state (thread 0): the next descriptor, loaded one chunk ahead,
    // and the liveness of the LP it belongs to
    Chunk nxt{};
    StLp plp;
    auto produce = [&](int j, int s) {   // chunk q0 + j into stage s
        const Chunk ch = nxt;
        if (q0 + j + 1 < q1) nxt = chunks[q0 + j + 1];
        if (ch.inst != plp.inst) st_load_lp<PRIMAL>(plp, b, ch.inst, it);
        st_issue<VT, PRIMAL>(ch, plp.live, stage0 + (size_t)s * Ly::kBytes, bar + s, b, src, pol);
    };
    // everything staged reads data written two or more launches back
    if (tid == 0 && q0 < q1) {
        nxt = chunks[q0];
        for (int s = 0; s < stages && q0 + s < q1; s++) produce(s, s);
    }
    pdl_wait();
    pdl_trigger();
    const double *__restrict__ g = PRIMAL ? b.y[src] : b.xsum;   // gathered vector
    StLp lp;
    const int n = q1 - q0;
    for (int i = 0; i < n; i++) {
        const int s = i % stages;
        const bool ok = mbar_wait(bar + s, (uint32_t)((i / stages) & 1));
        if (__syncthreads_or(!ok)) {
            // a stage never arrived: flag the LP, let the copies still in
            // flight land (each wait bounded again) and leave
            if (tid == 0) {
                b.S[chunks[q0 + i].inst].status = STALLED;
                const int issued = (i == 0) ? stages : i + stages - 1;   // chunks [0, issued) were issued
                for (int j = i; j < issued && j < n; j++) mbar_wait(bar + (j % stages), (uint32_t)((j / stages) & 1));
            }
            return;
        }
        // every thread is past chunk i-1: its stage can be refilled
        if (tid == 0 && i > 0 && i - 1 + stages < n) produce(i - 1 + stages, (i - 1) % stages);
        const unsigned char *sb = stage0 + (size_t)s * Ly::kBytes;
        const Chunk ch = *reinterpret_cast<const Chunk *>(sb);
        if (ch.inst != lp.inst) st_load_lp<PRIMAL>(lp, b, ch.inst, it);
        const int r = ch.r0 + tid;
        if (!lp.live || r >= ch.r1) continue;
        const StWindow<VT> w(ch);
        const int lr = r - w.r0a;
        const int *srp = reinterpret_cast<const int *>(sb + Ly::kRp);
        const int *sci = reinterpret_cast<const int *>(sb + Ly::kCi);
        const VT *sv = reinterpret_cast<const VT *>(sb + Ly::kVal);
        const double *vec = reinterpret_cast<const double *>(sb + Ly::kVec0);
        const int k0 = srp[r - w.rpa], k1 = srp[r + 1 - w.rpa];
        // the accumulator starts at -c (-q) and sums the row in entry order
        double acc = neg_bits(vec[1 * VS + lr]);
        const unsigned lanes = __activemask();
        for (int e = k0; __any_sync(lanes, e < k1); e += 4) {
            double gv[4];
            VT av[4];
#pragma unroll
            for (int u = 0; u < 4; u++)
                if (e + u < k1) { av[u] = sv[e + u - w.va]; gv[u] = g[sci[e + u - w.cia]]; }
            // an FMA step issues only if some lane of the warp needs it
#pragma unroll
            for (int u = 0; u < 4; u++) {
                if (!__any_sync(lanes, e + u < k1)) break;
                if (e + u < k1) acc = fma(widen(av[u]), gv[u], acc);
            }
        }
        const double zin = vec[lr];
        if (PRIMAL) {
            const long long *keys = reinterpret_cast<const long long *>(vec);
            const double xv = clip_keys(fma(lp.step, acc, zin), keys[2 * VS + lr], keys[3 * VS + lr]);
            const double xb = fma(2.0, xv, -zin);
            b.xsum[r] = xb;
            b.x[src ^ 1][r] = fma(lp.w, xb, lp.w1 * vec[4 * VS + lr]);
            if (lp.keep) b.xret[r] = xv;
        } else {
            double yv = fma(lp.step, acc, zin);
            if (r >= ch.aux) yv = nonneg(yv);
            b.y[src ^ 1][r] = fma(lp.w, fma(2.0, yv, -zin), lp.w1 * vec[2 * VS + lr]);
            if (lp.keep) b.yret[r] = yv;
        }
    }
}

}  // namespace dev
}  // namespace uc

#include "uc_block.cuh"

namespace uc {
namespace dev {

// ---------------------------------------------------------------------------
// shared-matrix ("lanes") iteration kernels (Halpern): K = 2 or 4 LPs with one
// scaled matrix, stored once; their vectors are interleaved, element j of lane
// r at j*K + r.  A row takes K/2 threads, each owning two lanes: its vector
// loads, stores and gathers are 16 bytes wide, the row's entries are read once
// for all lanes, and every thread carries two independent FMA chains.  Per
// lane the arithmetic is that of k_primal / k_dual, operation for operation.
// ---------------------------------------------------------------------------
template <int K>
struct LaneStep {   // per-lane data of one launch, shared by the CTA
    double step[K], w[K], w1[K];
    int live[K], keep[K];
};

template <int K, bool PRIMAL>
__device__ __forceinline__ void load_lane_steps(LaneStep<K> &L, const Bufs &b, int it) {
    const int r = threadIdx.x;
    if (r < K) {
        const Scalars *S = b.S + r;
        const int k = S->k_base + it;
        const bool live = S->status == RUNNING && k < S->max_iter;
        double w = 0.0, w1 = 0.0;
        if (live) halpern_weights(b, S, it, w, w1);
        L.live[r] = live;
        L.keep[r] = (it == S->n_eval - 1 || k == S->max_iter - 1);
        L.w[r] = w;
        L.w1[r] = w1;
        L.step[r] = PRIMAL ? S->tau : -S->sigma;
    }
    __syncthreads();
}

__device__ __forceinline__ void st_lanes(double *p, bool l0, bool l1, double v0, double v1) {
    if (l0 && l1) *reinterpret_cast<double2 *>(p) = make_double2(v0, v1);
    else if (l0) p[0] = v0;
    else if (l1) p[1] = v1;
}

template <typename VT, int K, int BS>
__global__ void __launch_bounds__(BS) k_primal_lanes(const Seg *__restrict__ segs, Bufs b, int it, int src) {
    constexpr int TPR = K / 2;   // threads per row
    __shared__ LaneStep<K> L;
    load_lane_steps<K, true>(L, b, it);
    const Seg sg = segs[blockIdx.x];
    const int j = sg.begin + (int)threadIdx.x / TPR;
    const int p = (int)threadIdx.x % TPR;
    const bool l0 = L.live[2 * p] != 0, l1 = L.live[2 * p + 1] != 0;
    if (j >= sg.end || !(l0 || l1)) { pdl_wait(); pdl_trigger(); return; }
    const VT *__restrict__ v = static_cast<const VT *>(b.AT_v);
    const size_t e = (size_t)j * K + 2 * p;   // this thread's first element
    // independent of the dual kernel that precedes this one
    const int k0 = __ldg(b.AT_rp + j), k1 = __ldg(b.AT_rp + j + 1);
    const double2 xin = ld_stream(reinterpret_cast<const double2 *>(b.x[src] + e));
    const longlong2 lk = ld_stream(reinterpret_cast<const longlong2 *>(b.lkey + e));
    const longlong2 uk = ld_stream(reinterpret_cast<const longlong2 *>(b.ukey + e));
    const double2 x0 = ld_stream(reinterpret_cast<const double2 *>(b.xa + e));
    int ci[kPre];
    double av[kPre];
#pragma unroll
    for (int q = 0; q < kPre; q++) {
        ci[q] = 0;
        av[q] = 0.0;
        if (k0 + q < k1) { ci[q] = ld_stream(b.AT_ci + k0 + q); av[q] = widen(ld_stream(v + k0 + q)); }
    }
    const double2 cc = ld_stream(reinterpret_cast<const double2 *>(b.c + e));
    double acc0 = neg_bits(cc.x), acc1 = neg_bits(cc.y);   // the accumulators end at A^T y - c
    pdl_wait();
    pdl_trigger();
    const double *__restrict__ y = b.y[src] + 2 * p;
    const unsigned lanes = __activemask();
#pragma unroll
    for (int q = 0; q < kPre; q++) {
        if (!__any_sync(lanes, k0 + q < k1)) break;
        if (k0 + q < k1) {
            const double2 g = *reinterpret_cast<const double2 *>(y + (size_t)ci[q] * K);
            acc0 = fma(av[q], g.x, acc0);
            acc1 = fma(av[q], g.y, acc1);
        }
    }
    for (int kk = k0 + kPre; kk < k1; kk++) {
        const double a = widen(ld_stream(v + kk));
        const double2 g = *reinterpret_cast<const double2 *>(y + (size_t)ld_stream(b.AT_ci + kk) * K);
        acc0 = fma(a, g.x, acc0);
        acc1 = fma(a, g.y, acc1);
    }
    double xv0 = 0.0, xv1 = 0.0, xb0 = 0.0, xb1 = 0.0, xn0 = 0.0, xn1 = 0.0;
    if (l0) {
        const int r = 2 * p;
        xv0 = clip_keys(fma(L.step[r], acc0, xin.x), lk.x, uk.x);
        xb0 = fma(2.0, xv0, -xin.x);
        xn0 = fma(L.w[r], xb0, L.w1[r] * x0.x);
    }
    if (l1) {
        const int r = 2 * p + 1;
        xv1 = clip_keys(fma(L.step[r], acc1, xin.y), lk.y, uk.y);
        xb1 = fma(2.0, xv1, -xin.y);
        xn1 = fma(L.w[r], xb1, L.w1[r] * x0.y);
    }
    st_lanes(b.xsum + e, l0, l1, xb0, xb1);
    st_lanes(b.x[src ^ 1] + e, l0, l1, xn0, xn1);
    st_lanes(b.xret + e, l0 && L.keep[2 * p], l1 && L.keep[2 * p + 1], xv0, xv1);
}

template <typename VT, int K, int BS>
__global__ void __launch_bounds__(BS) k_dual_lanes(const Seg *__restrict__ segs, Bufs b, int it, int src) {
    constexpr int TPR = K / 2;
    __shared__ LaneStep<K> L;
    load_lane_steps<K, false>(L, b, it);
    const Seg sg = segs[blockIdx.x];
    const int i = sg.begin + (int)threadIdx.x / TPR;
    const int p = (int)threadIdx.x % TPR;
    const bool l0 = L.live[2 * p] != 0, l1 = L.live[2 * p + 1] != 0;
    if (i >= sg.end || !(l0 || l1)) { pdl_wait(); pdl_trigger(); return; }
    const VT *__restrict__ v = static_cast<const VT *>(b.A_v);
    const size_t e = (size_t)i * K + 2 * p;
    const int k0 = __ldg(b.A_rp + i), k1 = __ldg(b.A_rp + i + 1);
    const double2 yin = ld_stream(reinterpret_cast<const double2 *>(b.y[src] + e));
    const double2 y0 = ld_stream(reinterpret_cast<const double2 *>(b.ya + e));
    int ci[kPre];
    double av[kPre];
#pragma unroll
    for (int q = 0; q < kPre; q++) {
        ci[q] = 0;
        av[q] = 0.0;
        if (k0 + q < k1) { ci[q] = ld_stream(b.A_ci + k0 + q); av[q] = widen(ld_stream(v + k0 + q)); }
    }
    const double2 qq = ld_stream(reinterpret_cast<const double2 *>(b.q + e));
    double acc0 = neg_bits(qq.x), acc1 = neg_bits(qq.y);   // the accumulators end at A x-bar - q
    pdl_wait();
    pdl_trigger();
    const double *__restrict__ xb = b.xsum + 2 * p;
    const unsigned lanes = __activemask();
#pragma unroll
    for (int q = 0; q < kPre; q++) {
        if (!__any_sync(lanes, k0 + q < k1)) break;
        if (k0 + q < k1) {
            const double2 g = *reinterpret_cast<const double2 *>(xb + (size_t)ci[q] * K);
            acc0 = fma(av[q], g.x, acc0);
            acc1 = fma(av[q], g.y, acc1);
        }
    }
    for (int kk = k0 + kPre; kk < k1; kk++) {
        const double a = widen(ld_stream(v + kk));
        const double2 g = *reinterpret_cast<const double2 *>(xb + (size_t)ld_stream(b.A_ci + kk) * K);
        acc0 = fma(a, g.x, acc0);
        acc1 = fma(a, g.y, acc1);
    }
    const bool ineq = i >= sg.aux;
    double yv0 = 0.0, yv1 = 0.0, yn0 = 0.0, yn1 = 0.0;
    if (l0) {
        const int r = 2 * p;
        yv0 = fma(L.step[r], acc0, yin.x);
        if (ineq) yv0 = nonneg(yv0);
        yn0 = fma(L.w[r], fma(2.0, yv0, -yin.x), L.w1[r] * y0.x);
    }
    if (l1) {
        const int r = 2 * p + 1;
        yv1 = fma(L.step[r], acc1, yin.y);
        if (ineq) yv1 = nonneg(yv1);
        yn1 = fma(L.w[r], fma(2.0, yv1, -yin.y), L.w1[r] * y0.y);
    }
    st_lanes(b.y[src ^ 1] + e, l0, l1, yn0, yn1);
    st_lanes(b.yret + e, l0 && L.keep[2 * p], l1 && L.keep[2 * p + 1], yv0, yv1);
}

// lane `lane` of the interleaved state <- its start point (x_init, y_init)
__global__ void k_lane_reset(Bufs b, const double *__restrict__ x_init, const double *__restrict__ y_init,
                             int n, int m, int K, int lane) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < (size_t)n) {
        const size_t e = t * K + lane;
        const double v = x_init[e];
        b.x[0][e] = v; b.x[1][e] = v; b.xa[e] = v; b.xret[e] = v; b.xsum[e] = 0.0;
    } else if (t < (size_t)n + m) {
        const size_t e = (t - n) * K + lane;
        const double v = y_init[e];
        b.y[0][e] = v; b.y[1][e] = v; b.ya[e] = v; b.yret[e] = v; b.ysum[e] = 0.0;
    }
}

// dst[t] <- src[t*K + lane] (gather = true) or dst[t*K + lane] <- src[t] (scatter)
__global__ void k_lane_copy(double *__restrict__ dst, const double *__restrict__ src, int count, int K, int lane,
                            int gather) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= count) return;
    if (gather) dst[t] = src[(size_t)t * K + lane];
    else dst[(size_t)t * K + lane] = src[t];
}

// ---------------------------------------------------------------------------
// evaluation: per-CTA FP64 partials of both candidates (fixed reduction order)
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool slot_is_max(int s) { return (s % kSlots) == RPU || (s % kSlots) == RDU; }

// Block reduction of an evaluation record with few FP64 instructions.  The 14
// sum slots go through a transposed warp reduction: at each of five exchange
// steps a lane keeps half of its remaining slots and adds its partner's copy,
// so every FP64 add is useful (16 adds per lane instead of 5 per slot); lanes
// 2s and 2s+1 end with the warp sum of slot s.  The 4 maxima of non-negative
// values use integer shuffles.  Warps are combined in a fixed order, so the
// result is deterministic.
__host__ __device__ constexpr int sum_slot(int i) {   // i in [0, 14)
    return (i < 7 ? 0 : kSlots) + ((i % 7) == 0 ? RP2 : (i % 7) == 1 ? QY : (i % 7) == 2 ? DY2 :
                                   (i % 7) == 3 ? RD2 : (i % 7) == 4 ? CX : (i % 7) == 5 ? BND : DX2);
}
__host__ __device__ constexpr int max_slot(int i) {   // i in [0, 4)
    return (i < 2 ? 0 : kSlots) + ((i & 1) ? RDU : RPU);
}

__device__ __forceinline__ void block_reduce_record(const double (&acc)[kPart], double *out) {
    __shared__ double sh[kThreads / 32][16];
    __shared__ long long shm[kThreads / 32][4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double v[16];
#pragma unroll
    for (int i = 0; i < 14; i++) v[i] = acc[sum_slot(i)];
    v[14] = 0.0;
    v[15] = 0.0;
#pragma unroll
    for (int half = 8, bit = 16; half >= 1; half >>= 1, bit >>= 1) {
        const bool up = (lane & bit) != 0;
#pragma unroll
        for (int i = 0; i < half; i++) {
            const double send = up ? v[i] : v[i + half];
            const double keep = up ? v[i + half] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
        }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
    if ((lane & 1) == 0) sh[warp][lane >> 1] = v[0];
#pragma unroll
    for (int i = 0; i < 4; i++) {
        long long m = __double_as_longlong(acc[max_slot(i)]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const long long other = __shfl_xor_sync(0xffffffffu, m, o);
            m = other > m ? other : m;
        }
        if (lane == 0) shm[warp][i] = m;
    }
    __syncthreads();
    if (threadIdx.x < 14) {
        double t = sh[0][threadIdx.x];
        for (int w = 1; w < kThreads / 32; w++) t += sh[w][threadIdx.x];
        out[sum_slot(threadIdx.x)] = t;
    } else if (threadIdx.x >= 32 && threadIdx.x < 36) {
        const int i = threadIdx.x - 32;
        long long m = shm[0][i];
        for (int w = 1; w < kThreads / 32; w++) m = shm[w][i] > m ? shm[w][i] : m;
        out[max_slot(i)] = __longlong_as_double(m);
    }
}

// Selections of the evaluation on the integer pipe (the kernel is FP64-bound):
// sign and finiteness from the bit pattern, max(v, 0) / min(v, 0) as a choice
// between v and 0.  Where they differ from fmax / fmin (a zero's sign) the
// value is only squared, taken absolutely or added to a sum, so the records
// are unchanged.
__device__ __forceinline__ bool is_neg(double v) { return __double_as_longlong(v) < 0; }
__device__ __forceinline__ bool is_fin(double v) {
    return (__double_as_longlong(v) & 0x7ff0000000000000LL) != 0x7ff0000000000000LL;
}
__device__ __forceinline__ double pos_part(double v) { return is_neg(v) ? 0.0 : v; }
__device__ __forceinline__ double neg_part(double v) { return is_neg(v) ? v : 0.0; }

// Terms that are exact zeros for a whole warp are skipped (the kernel is bound by
// the FP64 pipe): any_bits: some value is not a zero; differ: a - b is not an
// exact zero (two equal values that are not finite differ: inf - inf).
__device__ __forceinline__ bool any_bits(unsigned lanes, double v) { return __any_sync(lanes, (__double_as_longlong(v) << 1) != 0); }
__device__ __forceinline__ bool differ(double a, double b) { return __double_as_longlong(a) != __double_as_longlong(b) || !is_fin(a); }

// f(value, g[j], j) for entries k0, k0 + step, ... < k1 of a row, in order; the
// loads of four entries are in flight together (one after another they are the
// evaluation's time: 6 round trips to L2 for a row of three entries instead of 3)
template <typename VT, typename At, typename F>
__device__ __forceinline__ void each_entry(const int *__restrict__ ci, const VT *__restrict__ v, const double *g, At at,
                                           unsigned k, unsigned k1, int step, F f) {
    for (int left = (int)(k1 - k); left > 0; left -= 4 * step, k += 4 * step) {   // k1 may be close to 2^31
        size_t j[4];
        double a[4], gj[4];
#pragma unroll
        for (int q = 0; q < 4; q++)
            if (q * step < left) { j[q] = at(__ldg(ci + k + q * step)); a[q] = widen(__ldg(v + k + q * step)); }
#pragma unroll
        for (int q = 0; q < 4; q++) if (q * step < left) gj[q] = g[j[q]];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            if (q * step >= left) break;
            f(a[q], gj[q], j[q]);
        }
    }
}

// mode 0: the start point (candidate 0 only); mode 1: regular evaluation.
// Average variant: candidate 0 = current point, candidate 1 = average since the
// last restart.  Halpern variant: candidate 0 = the last map output
// (x_hat, y_hat); the record of candidate 1 only carries the fixed-point
// residual ||x_in - x_hat||^2 (slot DX2) and ||y_in - y_hat||^2 (slot DY2),
// x_in / y_in being the input of the last step (buffer 1, n_eval even).
// K > 1: shared-matrix session, vectors interleaved by lane; lane blockIdx.y.
template <typename VT, int K>
__global__ void __launch_bounds__(kThreads, 3) k_eval(const Seg *__restrict__ segs, Bufs b, int mode) {
    const Seg sg = segs[blockIdx.x];
    const int lane = (K == 1) ? 0 : (int)blockIdx.y;
    // a resident block kernel before this one has ended: the next one's tags differ from its tags
    if (mode == 1 && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *b.blk_seq += (unsigned)b.n_eval;
    const Scalars *S = b.S + ((K == 1) ? sg.inst : lane);
    auto at = [lane](int idx) { return (size_t)idx * K + lane; };
    double acc[kPart];
#pragma unroll
    for (int s = 0; s < kPart; s++) acc[s] = 0.0;
    const bool live = (mode == 0) ? (S->status == NEEDS_INIT)
                                  : (S->status == RUNNING && S->k_base + S->n_eval <= S->max_iter);
    if (live) {
        const bool halp = S->algo == ALG_HALPERN && mode == 1;
        const bool fpr = halp && S->metric != METRIC_KKT;   // fixed-point residual terms needed
        // the PDHG-norm residual also needs (y_in - y_hat).A (x_in - x_hat), summed
        // in candidate 1's CX slot (unused by the Halpern variant)
        const bool fprp = halp && S->metric == METRIC_FPRP;
        // infeasibility direction dy = y_hat - y_in: q.dy in slot QY, the bound part
        // of its objective in BND, the y_I < 0 and reduced-cost cone violations
        // (unscaled) as maxima in RPU and RDU, all of the second record
        const bool ray = halp && (S->evals + 1) % kInfeasEvery == 0;
        const bool avg = S->algo == ALG_AVERAGE && mode == 1;
        const double *x = halp ? b.xret : b.x[0];
        const double *y = halp ? b.yret : b.y[0];
        // average = sums / steps; with adaptive steps, sums / (sum of accepted
        // steps), or the current point when no step was accepted since the restart
        double inv_j = 0.0;
        const double *xav = b.xsum, *yav = b.ysum;
        if (avg && S->adaptive) {
            if (S->wsum > 0.0) inv_j = S->inv_wsum;
            else { inv_j = 1.0; xav = x; yav = y; }
        } else if (avg) {
            inv_j = S->inv_next;   // 1 / (j_base + n_eval)
        }
        const bool rows = (sg.aux & 1) == 0;
        const int eq_end = sg.aux >> 1;   // rows: first ">=" row
        if (rows) {
            const VT *__restrict__ v = static_cast<const VT *>(b.A_v);
            for (int i = sg.begin + threadIdx.x; i < sg.end; i += kThreads) {
                double ax0 = 0.0, ax1 = 0.0, axin = 0.0;
                each_entry(b.A_ci, v, x, at, __ldg(b.A_rp + i), __ldg(b.A_rp + i + 1), 1, [&](double a, double xj, size_t j) {
                    ax0 = fma(a, xj, ax0);
                    if (avg) ax1 = fma(a, xav[j] * inv_j, ax1);
                    if (fprp) axin = fma(a, b.x[1][j], axin);
                });
                const size_t ii = at(i);
                const double qi = b.q[ii], idr = b.inv_Dr[ii], yh = b.ya[ii];
                const bool ineq = i >= eq_end;
                double r0 = ax0 - qi;
                if (ineq && !is_neg(r0)) r0 = 0.0;
                const double y0 = y[ii];
                const unsigned lanes = __activemask();
                if (any_bits(lanes, r0)) {
                    acc[RP2] = fma(r0, r0, acc[RP2]);
                    acc[RPU] = nnmax(acc[RPU], fabs(r0) * idr);
                }
                if (__any_sync(lanes, (__double_as_longlong(qi) << 1) != 0 || !is_fin(y0))) acc[QY] = fma(qi, y0, acc[QY]);
                if (__any_sync(lanes, differ(y0, yh))) acc[DY2] = fma(y0 - yh, y0 - yh, acc[DY2]);
                if (avg) {
                    double r1 = ax1 - qi;
                    if (ineq && !is_neg(r1)) r1 = 0.0;
                    const double y1 = yav[ii] * inv_j;
                    acc[kSlots + RP2] += r1 * r1;
                    acc[kSlots + RPU] = nnmax(acc[kSlots + RPU], fabs(r1) * idr);
                    acc[kSlots + QY] += qi * y1;
                    acc[kSlots + DY2] += (y1 - yh) * (y1 - yh);
                } else if (fpr) {
                    const double d = b.y[1][ii] - y0;
                    acc[kSlots + DY2] += d * d;
                    if (fprp) acc[kSlots + CX] += d * (axin - ax0);
                }
                if (ray) {
                    const double dy = y0 - b.y[1][ii];
                    acc[kSlots + QY] += qi * dy;
                    if (ineq) acc[kSlots + RPU] = nnmax(acc[kSlots + RPU], (is_neg(dy) ? -dy : 0.0) * b.Dr[ii]);
                }
            }
        } else {
            const VT *__restrict__ v = static_cast<const VT *>(b.AT_v);
            // a slice of long columns (rpt = 0): a warp per column, lanes striding
            // over its entries, lane 0 accumulating the column's terms
            const bool lng = sg.rpt == 0;
            const int wl = threadIdx.x & 31;
            for (int j = lng ? sg.begin + (int)(threadIdx.x >> 5) : sg.begin + (int)threadIdx.x; j < sg.end;
                 j += lng ? sg.end - j : kThreads) {
                double t0 = 0.0, t1 = 0.0, tr = 0.0;
                const int e0 = b.AT_rp[j] + (lng ? wl : 0), e1 = b.AT_rp[j + 1], es = lng ? 32 : 1;
                each_entry(b.AT_ci, v, y, at, e0, e1, es, [&](double a, double yi, size_t i) {
                    t0 = fma(a, yi, t0);
                    if (avg) t1 = fma(a, yav[i] * inv_j, t1);
                    if (ray) tr = fma(a, yi - b.y[1][i], tr);
                });
                if (lng) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        t0 += __shfl_xor_sync(0xffffffffu, t0, o);
                        if (avg) t1 += __shfl_xor_sync(0xffffffffu, t1, o);
                        if (ray) tr += __shfl_xor_sync(0xffffffffu, tr, o);
                    }
                    if (wl != 0) break;
                }
                const size_t jj = at(j);
                const double cj = b.c[jj], lj = b.l[jj], uj = b.u[jj], idc = b.inv_Dc[jj], xh = b.xa[jj];
                const bool lf = is_fin(lj), uf = is_fin(uj);
                const double lam[2] = {cj - t0, cj - t1};
                const double xs[2] = {x[jj], avg ? xav[jj] * inv_j : 0.0};
#pragma unroll
                for (int cnd = 0; cnd < 2; cnd++) {
                    if (cnd == 1 && !avg) break;
                    const double lm = lam[cnd];
                    const double lp = (lf && uf) ? lm : lf ? pos_part(lm) : uf ? neg_part(lm) : 0.0;
                    const unsigned lanes = __activemask();
                    double *a = acc + cnd * kSlots;
                    if (__any_sync(lanes, differ(lm, lp))) {   // a boxed column has none
                        const double rd = lm - lp;
                        a[RD2] = fma(rd, rd, a[RD2]);
                        a[RDU] = nnmax(a[RDU], fabs(rd) * idc);
                    }
                    if (__any_sync(lanes, (__double_as_longlong(cj) << 1) != 0 || !is_fin(xs[cnd]))) a[CX] = fma(cj, xs[cnd], a[CX]);
                    const double bound = is_neg(lp) ? (uf ? uj : 0.0) : (lf ? lj : 0.0);
                    if (any_bits(lanes, bound)) a[BND] = fma(bound, lp, a[BND]);
                    if (__any_sync(lanes, differ(xs[cnd], xh))) a[DX2] = fma(xs[cnd] - xh, xs[cnd] - xh, a[DX2]);
                }
                if (fpr) {
                    const double d = b.x[1][jj] - x[jj];
                    acc[kSlots + DX2] += d * d;
                }
                if (ray) {   // reduced cost of the direction: lam = -A^T dy
                    const double lm = -tr;
                    const double lp = (lf && uf) ? lm : lf ? pos_part(lm) : uf ? neg_part(lm) : 0.0;
                    double bnd = 0.0;
                    if (lf) bnd += lj * pos_part(lp);
                    if (uf) bnd += uj * neg_part(lp);
                    acc[kSlots + BND] += bnd;
                    acc[kSlots + RDU] = nnmax(acc[kSlots + RDU], fabs(lm - lp) * idc);
                }
            }
        }
    }
    const size_t rec = (K == 1) ? blockIdx.x : (size_t)blockIdx.y * gridDim.x + blockIdx.x;
    block_reduce_record(acc, b.part + rec * kPart);
}

// ---------------------------------------------------------------------------
// reduction of the evaluation records: one CTA per (LP, slot), fixed order
// (FP64 adds spread over kPart CTAs per LP instead of one)
// ---------------------------------------------------------------------------
struct InstRange { int eval_begin, eval_end; };

__global__ void __launch_bounds__(kThreads) k_reduce(const InstRange *__restrict__ ranges, Bufs b, int mode) {
    const int inst = blockIdx.x / kPart, slot = blockIdx.x % kPart;
    const Scalars *S = b.S + inst;
    const bool live = (mode == 0) ? (S->status == NEEDS_INIT) : (S->status == RUNNING);
    if (!live) return;
    const InstRange r = ranges[inst];
    const bool mx = slot_is_max(slot);
    double acc = 0.0;
    for (int blk = r.eval_begin + threadIdx.x; blk < r.eval_end; blk += kThreads) {
        const double p = b.part[(size_t)blk * kPart + slot];
        acc = mx ? nnmax(acc, p) : acc + p;
    }
    __shared__ double sh[kThreads];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int h = kThreads / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) sh[threadIdx.x] = mx ? nnmax(sh[threadIdx.x], sh[threadIdx.x + h]) : sh[threadIdx.x] + sh[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) b.red[(size_t)inst * kPart + slot] = sh[0];
}

// ---------------------------------------------------------------------------
// scalar controller: one warp per LP
// ---------------------------------------------------------------------------
// Every FP64 quotient, root, logarithm and exponential is a long chain of FP64
// instructions, and one thread takes them one after another: 10 us of the 35 us
// an evaluation takes on the 30-bus LP.  Here the lanes of a warp take those that
// do not depend on one another side by side (one instruction stream), the
// scalars are read by all lanes and written by the first.
__device__ double kkt_w(double rp2, double rd2, double gap, double w) {
    return sqrt(w * w * rp2 + rd2 / (w * w) + gap * gap);
}

__device__ __forceinline__ double lane_val(double v, int lane) { return __shfl_sync(0xffffffffu, v, lane); }

// Primal weight at a restart from the epoch's movement dx (primal), dy (dual).
// The error e = ln(omega dx / dy) is zero when the weighted movements
// omega dx^2 and dy^2 / omega balance.  The update is a PID controller on ln
// omega: ln omega <- ln omega - (kp e + ki sum(e) + kd (e - e_prev)).  PDLP's
// rule, omega <- exp(0.5 ln(dy/dx) + 0.5 ln omega), is the proportional part
// with kp = 0.5 and is computed in that form.  omega is kept when dx or dy is
// at most 1e-10.  Called by a warp; isum, eprev and has are the controller's
// state, which the caller stores.
__device__ __forceinline__ double primal_weight(const Scalars *S, double w, double dx, double dy, double &isum, double &eprev,
                                                int &has) {
    if (!(dx > 1e-10 && dy > 1e-10)) return w;
    const bool odd = threadIdx.x & 1;
    if (S->pw_kp == 0.5 && S->pw_ki == 0.0 && S->pw_kd == 0.0) {
        const double lg = log(odd ? w : dy / dx);
        return exp(0.5 * lane_val(lg, 0) + 0.5 * lane_val(lg, 1));
    }
    const double lg = log(odd ? w : w * dx / dy);
    const double e = lane_val(lg, 0);
    isum += e;
    const double de = has ? e - eprev : 0.0;
    eprev = e;
    has = 1;
    return exp(lane_val(lg, 1) - (S->pw_kp * e + S->pw_ki * isum + S->pw_kd * de));
}

// Residual-balance guard: a larger omega is a larger dual step, which works on
// primal infeasibility, and a smaller one the reverse.  The controller's new
// weight wn is dropped (omega kept) when it moves against the balance of the
// relative residuals of the restart point by more than the factor kappa.
__device__ double guard_weight(const Scalars *S, double w, double wn, double rel_p, double rel_d) {
    const double kap = S->pw_guard;
    if (kap > 0.0 && ((wn < w && rel_p > kap * rel_d) || (wn > w && rel_d > kap * rel_p))) return w;
    return wn;
}

// the evaluation's decision for LP `inst`, by a whole warp
__device__ void control_lp(const Bufs &b, int mode, int inst) {
    Scalars *S = b.S + inst;
    const int lane = threadIdx.x & 31;
    const bool first = lane == 0;
    const int status = S->status;
    const double *T = b.red + (size_t)inst * kPart;
    const double w = S->omega;
    __syncwarp();
    if (first) S->action = ACT_NONE;
    if (mode == 0 ? status != NEEDS_INIT : status != RUNNING) return;
    // lanes 4 c .. 4 c + 3: the quotients of candidate c
    const double *Ta = T + (lane >> 2 & 1) * kSlots;
    double num, den;
    {
        const double po = Ta[CX], dob = Ta[QY] + Ta[BND], g = po - dob;
        const int q = lane & 3;
        num = q == 0 ? Ta[RPU] : q == 1 ? Ta[RDU] : q == 2 ? fabs(g) : Ta[RD2];
        den = q == 0 ? 1.0 + S->q_inf : q == 1 ? 1.0 + S->c_inf : q == 2 ? 1.0 + fabs(po) + fabs(dob) : w * w;
        num = num / den;
        den = sqrt(w * w * Ta[RP2] + num + g * g);   // the weighted KKT error where q = 3
    }
    double K[2], rel[2][3], gap[2], pobj[2], dobj[2];
#pragma unroll
    for (int cnd = 0; cnd < 2; cnd++) {
        const double *a = T + cnd * kSlots;
        pobj[cnd] = a[CX];
        dobj[cnd] = a[QY] + a[BND];
        gap[cnd] = pobj[cnd] - dobj[cnd];
#pragma unroll
        for (int q = 0; q < 3; q++) rel[cnd][q] = lane_val(num, 4 * cnd + q);
        K[cnd] = lane_val(den, 4 * cnd + 3);
    }
    const int algo = S->algo, metric = S->metric;
    auto report = [&](int cnd) {
        S->rel_p = rel[cnd][0]; S->rel_d = rel[cnd][1]; S->rel_g = rel[cnd][2];
        S->abs_p = T[cnd * kSlots + RPU]; S->pobj = pobj[cnd]; S->dobj = dobj[cnd];
    };
    auto stop = [&](int st) { S->status = st; b.status[inst] = st; };
    if (mode == 0) {                     // initial anchor (no residual yet for the fixed-point metric)
        if (!first) return;
        S->kkt_anchor = (algo == ALG_HALPERN && metric != METRIC_KKT) ? INFINITY : K[0];
        S->kkt_prev = INFINITY;
        report(0);
        stop(isfinite(K[0]) ? RUNNING : NUMERIC);
        return;
    }
    const int n_eval = S->n_eval, max_iter = S->max_iter, k = S->k_base + n_eval, j = S->j_base + n_eval;
    if (k > max_iter) {                  // partial block: limit reached inside it
        if (first) stop(ITER_LIMIT);
        return;
    }
    const int evals = S->evals + 1;
    const double anchor = S->kkt_anchor, prev = S->kkt_prev, eta = S->eta, tol = S->tol, stop_abs = S->stop_abs;
    const double ad_eta = S->ad_eta;
    double isum = S->pw_isum, eprev = S->pw_eprev;
    int has = S->pw_has;
    __syncwarp();
    if (first) {
        S->evals = evals;
        S->inv_j = S->adaptive ? (S->wsum > 0.0 ? S->inv_wsum : 0.0) : S->inv_next;
        S->k_base = k;
    }
    if (algo == ALG_HALPERN) {
        // candidate 0 = last map output; fixed-point residual terms in the second record
        const double fx2 = T[kSlots + DX2], fy2 = T[kSlots + DY2];
        if (!isfinite(K[0]) || !isfinite(fx2) || !isfinite(fy2)) {
            if (first) stop(NUMERIC);
            return;
        }
        if (first) report(0);
        if (stop_abs > 0.0 ? (T[RPU] <= stop_abs) : (fmax(rel[0][0], fmax(rel[0][1], rel[0][2])) <= tol)) {
            if (first) { stop(OPTIMAL); S->which = 0; }
            return;
        }
        if (evals % kInfeasEvery == 0) {
            const double obj = T[kSlots + QY] + T[kSlots + BND];
            const double viol = fmax(T[kSlots + RPU], T[kSlots + RDU]);
            if (obj > 0.0 && viol <= kInfeasEps * obj) {
                if (first) stop(INFEASIBLE);
                return;
            }
        }
        const double cross = (metric == METRIC_FPRP) ? T[kSlots + CX] : 0.0;
        const double r = (metric == METRIC_KKT) ? K[0] : sqrt(fmax(w * fx2 + fy2 / w - 2.0 * eta * cross, 0.0));
        const bool restart = (r <= 0.2 * anchor) || (r <= 0.8 * anchor && r > prev) || ((double)j >= 0.36 * (double)k);
        if (restart) {
            const double root = sqrt(T[(lane & 1) ? DY2 : DX2]);
            const double dx = lane_val(root, 0), dy = lane_val(root, 1);
            const double wn = guard_weight(S, w, primal_weight(S, w, dx, dy, isum, eprev, has), rel[0][0], rel[0][1]);
            // tau and the anchor's quotient side by side
            const double quo = ((lane & 1) ? (metric == METRIC_KKT ? T[RD2] : fy2) : eta) /
                               ((lane & 1) && metric == METRIC_KKT ? wn * wn : wn);
            const double tau = lane_val(quo, 0), part = lane_val(quo, 1);
            const double an = metric == METRIC_KKT ? sqrt(wn * wn * T[RP2] + part + gap[0] * gap[0])
                                                   : sqrt(fmax(wn * fx2 + part - 2.0 * eta * cross, 0.0));
            if (first) {
                S->omega = wn;
                S->pw_isum = isum; S->pw_eprev = eprev; S->pw_has = has;
                S->kkt_anchor = an;
                S->kkt_prev = INFINITY;
                S->j_base = 0;
                S->restarts += 1;
                S->tau = tau;
                S->sigma = eta * wn;
                S->action = ACT_RESTART;
            }
        } else if (first) {
            S->kkt_prev = r;
            S->j_base = j;
        }
        if (first && k >= max_iter) stop(ITER_LIMIT);
        return;
    }
    if (!isfinite(K[0]) || !isfinite(K[1])) {
        if (first) stop(NUMERIC);
        return;
    }
#pragma unroll
    for (int cnd = 0; cnd < 2; cnd++) {
        const double mx = fmax(rel[cnd][0], fmax(rel[cnd][1], rel[cnd][2]));
        if (mx <= tol) {
            if (first) { S->which = cnd; S->action = ACT_FINISH; report(cnd); stop(OPTIMAL); }
            return;
        }
    }
    if (first) report(0);
    const int cand = (K[1] < K[0]) ? 1 : 0;
    const double kc = cand ? K[1] : K[0];
    const bool restart = (kc <= 0.2 * anchor) || (kc <= 0.8 * anchor && kc > prev) || ((double)j >= 0.36 * (double)k);
    if (restart) {
        const double *a = T + cand * kSlots;
        const double root = sqrt(a[(lane & 1) ? DY2 : DX2]);
        const double dx = lane_val(root, 0), dy = lane_val(root, 1);
        const double wn = primal_weight(S, w, dx, dy, isum, eprev, has);
        const double quo = ((lane & 3) == 0 ? eta : (lane & 3) == 1 ? a[RD2] : ad_eta) / ((lane & 3) == 1 ? wn * wn : wn);
        const double tau = lane_val(quo, 0), part = lane_val(quo, 1), ad_tau = lane_val(quo, 2);
        const double g = cand ? gap[1] : gap[0];
        const double an = sqrt(wn * wn * a[RP2] + part + g * g);
        if (first) {
            S->omega = wn;
            S->pw_isum = isum; S->pw_eprev = eprev; S->pw_has = has;
            S->kkt_anchor = an;
            S->kkt_prev = INFINITY;
            S->j_base = 0;
            S->restarts += 1;
            S->tau = tau;
            S->sigma = eta * wn;
            S->cand = cand;
            S->wsum = 0.0;
            S->inv_wsum = 0.0;
            S->ad_tau = ad_tau;
            S->ad_sigma = ad_eta * wn;
            S->action = ACT_RESTART;
        }
    } else if (first) {
        S->kkt_prev = kc;
        S->j_base = j;
    }
    if (!first) return;
    S->inv_next = 1.0 / (double)((restart ? 0 : j) + n_eval);
    if (k >= max_iter) stop(ITER_LIMIT);
}

constexpr int kControlThreads = 128;   // four LPs per CTA
__global__ void __launch_bounds__(kControlThreads) k_control(Bufs b, int mode, int k_lps) {
    const int inst = (int)(blockIdx.x * kControlThreads + threadIdx.x) >> 5;
    if (inst < k_lps) control_lp(b, mode, inst);
}

// Average variant: restart (current <- candidate, anchor <- candidate,
// sums <- 0) or finish (returned point <- chosen candidate).  Halpern variant:
// restart (current <- map output, anchor <- map output).
// K > 1: shared-matrix session, lane blockIdx.y, vectors interleaved by lane.
template <int BS, int K>
__global__ void __launch_bounds__(BS) k_apply(const Seg *__restrict__ segs, int ncol_blocks, Bufs b) {
    const Seg sg = segs[blockIdx.x];
    const int lane = (K == 1) ? 0 : (int)blockIdx.y;
    const Scalars *S = b.S + ((K == 1) ? sg.inst : lane);
    const int act = S->action;
    if (act == ACT_NONE) return;
    for (int t = 0; t < sg.rpt; t++) {
    const int row = sg.begin + t * BS + threadIdx.x;
    if (row >= sg.end) return;
    const size_t idx = (size_t)row * K + lane;
    const bool col = blockIdx.x < (unsigned)ncol_blocks;
    double *cur = col ? b.x[0] : b.y[0];
    double *sum = col ? b.xsum : b.ysum;
    double *anc = col ? b.xa : b.ya;
    double *ret = col ? b.xret : b.yret;
    if (S->algo == ALG_HALPERN) {
        const double v = ret[idx];
        cur[idx] = v;
        anc[idx] = v;
        continue;
    }
    const double avg = sum[idx] * S->inv_j;
    if (act == ACT_FINISH) {
        ret[idx] = S->which ? avg : cur[idx];
        continue;
    }
    const double v = S->cand ? avg : cur[idx];
    cur[idx] = v;
    anc[idx] = v;
    sum[idx] = 0.0;
    }
}

// ---------------------------------------------------------------------------
// adaptive step size (PDLP, averaging variant; sessions of one LP)
// ---------------------------------------------------------------------------
// Every iteration is an attempt with the trial step eta = S->ad_eta:
//   k_ad_primal   x' = clip(x - (eta/omega)(c - A^T y), l, u) into the other
//                 buffer; per CTA: sum (x' - x)^2
//   k_ad_dual     y' = y + eta omega (q - A (2x' - x)), y'_I >= 0, into the
//                 other buffer; A (x' - x) from the same gathers; per CTA:
//                 sum (y' - y)^2 and sum (y' - y) (A (x' - x))_i
//   k_ad_decide   eta_bar = (omega |dx|^2 + |dy|^2 / omega) / (2 |dy^T A dx|);
//                 accepted when eta <= eta_bar (the current buffer flips and
//                 the step enters the weight sum); next trial
//                 min((1 - (a+2)^-0.3) eta_bar, (1 + (a+2)^-0.6) eta)
// An accepted step enters the running sums (+= eta * the accepted point) one
// kernel later: the next attempt's primal and dual kernels read that point as
// their input anyway, so they add it (S->ad_w holds the pending weight, 0 after
// a rejection).  Before each evaluation, k_ad_norm adds the last pending
// weight and moves the current iterate to buffer 0, so the evaluation, control
// and restart kernels of the averaging variant apply unchanged.  The kernels are plain one-thread-per-row loops: the option is
// for parity with the published method, not tuned.
constexpr int kAdThreads = 256;

__device__ __forceinline__ bool ad_live(const Scalars *S, int it) {
    return S->status == RUNNING && S->k_base + it < S->max_iter;
}

// fixed-order CTA sum of NV values per thread into out[0..NV)
template <int NV>
__device__ __forceinline__ void ad_block_sum(double (&v)[NV], double *out) {
    __shared__ double sh[kAdThreads / 32][NV];
#pragma unroll
    for (int q = 0; q < NV; q++) {
        double t = v[q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5][q] = t;
    }
    __syncthreads();
    if (threadIdx.x < NV) {
        double t = sh[0][threadIdx.x];
        for (int w = 1; w < kAdThreads / 32; w++) t += sh[w][threadIdx.x];
        out[threadIdx.x] = t;
    }
}

template <typename VT>
__global__ void __launch_bounds__(kAdThreads) k_ad_primal(Bufs b, int n, int it) {
    const Scalars *S = b.S;
    if (!ad_live(S, it)) return;
    const int src = S->ad_src;
    const double tau = S->ad_tau, w = S->ad_w;
    const VT *__restrict__ v = static_cast<const VT *>(b.AT_v);
    const double *__restrict__ y = b.y[src];
    const int j = blockIdx.x * kAdThreads + threadIdx.x;
    double d2[1] = {0.0};
    if (j < n) {
        const int k0 = __ldg(b.AT_rp + j), k1 = __ldg(b.AT_rp + j + 1);
        const double xin = b.x[src][j];
        double acc = neg_bits(ld_stream(b.c + j));   // ends at A^T y - c
        for (int k = k0; k < k1; k++) acc = fma(widen(ld_stream(v + k)), y[ld_stream(b.AT_ci + k)], acc);
        if (w != 0.0) b.xsum[j] = fma(w, xin, b.xsum[j]);   // the last accepted step
        const double xv = fmin(fmax(fma(tau, acc, xin), ld_stream(b.l + j)), ld_stream(b.u + j));
        b.x[src ^ 1][j] = xv;
        const double d = xv - xin;
        d2[0] = d * d;
    }
    ad_block_sum<1>(d2, b.adp + blockIdx.x);
}

template <typename VT>
__global__ void __launch_bounds__(kAdThreads) k_ad_dual(Bufs b, int m, int m_eq, int it, int nbp) {
    const Scalars *S = b.S;
    if (!ad_live(S, it)) return;
    const int src = S->ad_src;
    const double sigma = S->ad_sigma, w = S->ad_w;
    const VT *__restrict__ v = static_cast<const VT *>(b.A_v);
    const double *__restrict__ xn = b.x[src ^ 1];
    const double *__restrict__ xo = b.x[src];
    const int i = blockIdx.x * kAdThreads + threadIdx.x;
    double r[2] = {0.0, 0.0};
    if (i < m) {
        const int k0 = __ldg(b.A_rp + i), k1 = __ldg(b.A_rp + i + 1);
        const double yin = b.y[src][i];
        double acc = neg_bits(ld_stream(b.q + i));   // ends at A x-bar - q
        double adx = 0.0;                   // (A (x' - x))_i
        for (int k = k0; k < k1; k++) {
            const int j = ld_stream(b.A_ci + k);
            const double a = widen(ld_stream(v + k));
            acc = fma(a, fma(2.0, xn[j], -xo[j]), acc);
            adx = fma(a, xn[j] - xo[j], adx);
        }
        if (w != 0.0) b.ysum[i] = fma(w, yin, b.ysum[i]);   // the last accepted step
        double yv = fma(-sigma, acc, yin);
        if (i >= m_eq) yv = fmax(yv, 0.0);
        b.y[src ^ 1][i] = yv;
        const double dy = yv - yin;
        r[0] = dy * dy;
        r[1] = dy * adx;
    }
    ad_block_sum<2>(r, b.adp + nbp + 2 * (size_t)blockIdx.x);
}

// one CTA: the attempt's sums in a fixed order (strided partials per thread,
// then warp shuffles, then the 32 warp sums), then the acceptance test
__global__ void __launch_bounds__(1024) k_ad_decide(Bufs b, int nbp, int nbd, int it) {
    Scalars *S = b.S;
    if (!ad_live(S, it)) return;
    double v[3] = {0.0, 0.0, 0.0};
    for (int p = threadIdx.x; p < nbp; p += 1024) v[0] += b.adp[p];
    for (int p = threadIdx.x; p < nbd; p += 1024) {
        v[1] += b.adp[nbp + 2 * p];
        v[2] += b.adp[nbp + 2 * p + 1];
    }
    __shared__ double sh[32][3];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < 3; q++) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
        if (lane == 0) sh[warp][q] = v[q];
    }
    __syncthreads();
    if (warp != 0) return;
#pragma unroll
    for (int q = 0; q < 3; q++) {
        v[q] = sh[lane][q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
    }
    if (lane != 0) return;
    const double om = S->omega, eta = S->ad_eta;
    const double movement = om * v[0] + v[1] / om;
    const double interaction = fabs(v[2]);
    const double eta_bar = interaction > 0.0 ? movement / (2.0 * interaction) : INFINITY;
    const int a = S->k_base + it;   // attempt number (0-based)
    const double eta_next = fmin(b.adS[a] * eta_bar, b.adG[a] * eta);
    if (eta <= eta_bar) {
        S->ad_src ^= 1;
        S->ad_w = eta;
        S->wsum += eta;
        S->inv_wsum = 1.0 / S->wsum;
        S->ad_acc += 1;
    } else {
        S->ad_w = 0.0;
    }
    S->ad_eta = eta_next;
    S->ad_tau = eta_next / om;
    S->ad_sigma = eta_next * om;
}

// before an evaluation: the pending accepted step into the sums, and the
// current iterate to buffer 0 ...
__global__ void k_ad_norm(Bufs b, int n, int m) {
    const Scalars *S = b.S;
    const double w = S->ad_w;
    const int cur = S->ad_src;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) {
        const double v = b.x[cur][e];
        if (w != 0.0) b.xsum[e] = fma(w, v, b.xsum[e]);
        if (cur == 1) b.x[0][e] = v;
    } else if (e < n + m) {
        const double v = b.y[cur][e - n];
        if (w != 0.0) b.ysum[e - n] = fma(w, v, b.ysum[e - n]);
        if (cur == 1) b.y[0][e - n] = v;
    }
}
// ... and then the buffer index and the pending weight to 0
__global__ void k_ad_src0(Bufs b) {
    b.S->ad_src = 0;
    b.S->ad_w = 0.0;
}

// ---------------------------------------------------------------------------
// host orchestration: a device-resident session of k LPs
// ---------------------------------------------------------------------------
#define UC_CUDA(call)                                                                  \
    do {                                                                               \
        cudaError_t e_ = (call);                                                       \
        if (e_ != cudaSuccess) {                                                       \
            set_error("%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, \
                      __LINE__);                                                       \
            return UC_ECUDA;                                                           \
        }                                                                              \
    } while (0)

static size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

struct Layout {
    // uploaded once
    size_t A_rp, A_ci, A_v, AT_rp, AT_ci, AT_v, segs_p, segs_d, segs_e, segs_a, ranges;
    size_t W, W1, adS, adG;
    // per-LP data (replaced by update_lp)
    size_t c, l, u, Dc, q, Dr, inv_Dc, inv_Dr, lkey, ukey, x_init, y_init, S_init;
    // working state
    size_t x0, x1, y0, y1, xsum, ysum, xa, ya, xret, yret, part, red, S, status, adp;
    // staged kernels: chunk lists and per-CTA ranges
    size_t chunks_p, chunks_d, ctas_p, ctas_d;
    // period-strided groups: k per group and slot records (row kernels)
    size_t A_sk, AT_sk, A_sl, AT_sl;
    // resident block kernel: tiles, their split over warps, tagged vectors, iteration count, timing stamps
    size_t tiles, warps, image, xt, yt, blk_seq, stamp;
    // lanes sessions: contiguous staging for one LP's vectors (4 (n + m) doubles:
    // the seven vectors a result may download)
    size_t lane_stage;
    size_t upload_end, total;
};

}  // namespace dev
}  // namespace uc

struct uc_session {
    int k = 0, vb = 64;
    int cta = 128;                // rows (= threads) per CTA of the row kernels
    bool pdl = true;              // programmatic dependent launch between iteration kernels
    cudaError_t launch_err = cudaSuccess;
    int algo = 0;                 // ALG_HALPERN / ALG_AVERAGE (all LPs of a session)
    bool adaptive = false;        // adaptive step size (averaging variant, one LP)
    size_t vs = 8;
    uc_solve_opts o{};
    cudaStream_t s = nullptr;
    bool own_stream = false;
    std::vector<std::shared_ptr<const uc::PsData>> P;    // LPs in their own (natural) order
    // device views at creation: rows/columns reordered (later LPs of a slot have the
    // matrix and keep the order; their vectors are P's)
    std::vector<std::shared_ptr<const uc::PsData>> Pd;
    std::vector<std::vector<int32_t>> prow, pcol;        // device position -> natural index
    bool reorder = true;
    std::vector<int64_t> roff, coff, zoff;
    int64_t M = 0, N = 0, Z = 0;
    int n_sp = 0, n_sd = 0, n_se = 0, n_sa = 0;
    int n_sac = 0;   // column blocks at the head of the apply table
    uc::dev::Layout L{};
    char *D = nullptr;
    size_t bytes = 0;
    uc::dev::Bufs b{};
    const uc::dev::Seg *dsp = nullptr, *dsd = nullptr, *dse = nullptr, *dsa = nullptr;
    const uc::dev::InstRange *drg = nullptr;
    std::vector<uc::dev::Scalars> S_init;
    cudaGraph_t graph[2] = {nullptr, nullptr};
    cudaGraphExec_t exec[2] = {nullptr, nullptr};
    cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};
    cudaEvent_t tev[2][3] = {{nullptr, nullptr, nullptr}, {nullptr, nullptr, nullptr}};
    int *h_status = nullptr;      // pinned [k]
    std::vector<char> active;     // LPs reset since their last result
    std::vector<int> rpt;         // rows per thread of each LP's iteration CTAs
    std::vector<int> m_eq;        // equality rows of each LP
    std::vector<char> tabled;     // LPs whose CTAs are in the current tables and graph
    int cap_sp = 0, cap_sd = 0, cap_se = 0, cap_sa = 0;
    // shared-matrix ("lanes") sessions: K LPs with one scaled matrix, stored
    // once, vectors interleaved (element j of LP r at j*K + r); K = 1 otherwise,
    // also where the resident kernel takes the LPs one after another
    int K = 1;
    int64_t Mr = 0, Nr = 0;       // rows of A and of A^T as stored
    // primal feasibility polishing in progress: LPs reset now stop on this
    // absolute violation (0: the relative KKT test)
    double polish_tol = 0.0;
    // period-strided 16-row groups read from slot records (row kernels, K = 1)
    bool strided = false;
    int64_t strided_rows_A = 0, strided_rows_AT = 0;
    // resident block kernel: possible for this session; used by the current tables
    bool block_able = false, block = false;
    int sms = 0, blk_smem_max = 0;          // SMs, shared memory per CTA
    int blk_ctas = 0, blk_threads = 0, blk_smem = 0;
    int64_t blk_image = 0;                  // bytes of the tables' image
    uc::dev::BlockPlan plan{.polls = uc::dev::kBlockPolls};
    std::vector<std::array<std::vector<uc::dev::BlockTile>, 2>> cut;   // each LP's tiles, dual and primal (plan_block)
    unsigned long long *h_stamp = nullptr;   // pinned [2][2]: timed iteration's bounds of each graph
    unsigned long long last_stamp = 0;       // start of the iteration counted last
    double *h_vec = nullptr;      // pinned: an LP's vectors on their way to the device (update_lp)
    // staged iteration kernels
    bool staged = false;
    int stages = 4;
    int smem_p = 0, smem_d = 0;   // dynamic shared memory per CTA
    int gmax_p = 0, gmax_d = 0;   // resident CTAs on the device
    int g_p = 0, g_d = 0;         // CTAs of the current tables
    int cap_cp = 0, cap_cd = 0;   // chunk capacities
    const uc::dev::Chunk *dcp = nullptr, *dcd = nullptr;
    const int *dgp = nullptr, *dgd = nullptr;
    int retables = 0;
    double tp_sum = 0.0, td_sum = 0.0;
    int timed = 0;
    long long launches = 0;
    double upload_ms = 0.0, last_run_ms = 0.0;
    int host_status = UC_OK;      // UC_ECANCELLED / UC_ETIMEOUT of the last run
    long long h2d = 0;            // bytes uploaded (create, update_lp, set_start)
    long long polls = 0;          // replays whose status was copied back

    ~uc_session() {
        if (s) cudaStreamSynchronize(s);
        for (auto e : exec) if (e) cudaGraphExecDestroy(e);
        for (auto g : graph) if (g) cudaGraphDestroy(g);
        for (auto e : ev) if (e) cudaEventDestroy(e);
        for (auto &row : tev) for (auto e : row) if (e) cudaEventDestroy(e);
        if (h_status) cudaFreeHost(h_status);
        if (h_stamp) cudaFreeHost(h_stamp);
        if (h_vec) cudaFreeHost(h_vec);
        if (D) {
            if (o.free) o.free(D, bytes, (void *)s, o.alloc_ctx);
            else cudaFreeAsync(D, s);
        }
        if (own_stream && s) { cudaStreamSynchronize(s); cudaStreamDestroy(s); }
    }
};

namespace uc {
namespace dev {

template <typename T>
static void put(std::vector<char> &st, size_t off, const T *src, size_t count) {
    if (count) std::memcpy(st.data() + off, src, count * sizeof(T));
}

// Device view of an LP.  Rows and columns are put in entity-major order: by
// (kind, unit / bus / line, period) of the raw LP they come from, equality
// rows first.  Consecutive rows are then one constraint of one unit, bus or
// line in consecutive periods, whose entries point at one variable of one
// entity in consecutive periods, which the device stores consecutively too:
// a warp's gathers read a few contiguous sectors instead of one sector per
// thread.  Warps issue as many FMA iterations as their longest row, so within
// windows of kOrderWindow rows of that order the rows are then sorted by
// decreasing length (stable).  Columns get the same treatment with their A^T
// row length.  Each row keeps its entries in their original order, so every
// dot product sums in the same order as in the natural layout, except that the
// columns with more than kLongRow entries go last and a warp sums each of them
// (primal_long).
constexpr int kOrderWindow = 1024;

static void window_order(const std::vector<int32_t> &rp, const std::vector<int32_t> &base, std::vector<int32_t> &out) {
    for (size_t w0 = 0; w0 < base.size(); w0 += kOrderWindow) {
        const size_t w1 = std::min(base.size(), w0 + (size_t)kOrderWindow);
        const size_t o = out.size();
        out.insert(out.end(), base.begin() + w0, base.begin() + w1);
        std::stable_sort(out.begin() + o, out.end(), [&](int32_t a, int32_t b) {
            return rp[a + 1] - rp[a] > rp[b + 1] - rp[b];
        });
    }
}

// [begin, end) sorted by the (kind, entity, period) of the raw row or column
// each maps to; natural order when the raw labels are missing
static std::vector<int32_t> entity_order(int begin, int end, const std::vector<int32_t> &map,
                                         const std::vector<int8_t> &kind, const std::vector<int32_t> &ent,
                                         const std::vector<int32_t> &per) {
    std::vector<int32_t> o;
    o.reserve(end - begin);
    for (int r = begin; r < end; r++) o.push_back(r);
    const size_t nraw = kind.size();
    bool ok = ent.size() == nraw && per.size() == nraw && (int64_t)map.size() >= end;
    for (int r = begin; ok && r < end; r++) ok = map[r] >= 0 && (size_t)map[r] < nraw;
    if (!ok) return o;
    // the (kind, entity, period) label packed into one ordered 64-bit key (kind:
    // 8 bits, entity: 32, period: 24); labels of one LP are distinct, so sorting
    // (key, index) pairs gives the order of a stable sort by label
    bool packable = true;
    std::vector<std::pair<uint64_t, int32_t>> kv;
    kv.reserve(o.size());
    for (int32_t r : o) {
        const int32_t rr = map[r];
        packable &= kind[rr] >= 0 && ent[rr] >= 0 && per[rr] >= 0 && per[rr] < (1 << 24);
        kv.push_back({((uint64_t)(uint8_t)kind[rr] << 56) | ((uint64_t)(uint32_t)ent[rr] << 24) | (uint64_t)per[rr], r});
    }
    if (packable) {
        std::sort(kv.begin(), kv.end());
        bool distinct = true;
        for (size_t t = 1; t < kv.size() && distinct; t++) distinct = kv[t].first != kv[t - 1].first;
        if (distinct) {
            for (size_t t = 0; t < kv.size(); t++) o[t] = kv[t].second;
            return o;
        }
    }
    std::stable_sort(o.begin(), o.end(), [&](int32_t a, int32_t b) {
        const int32_t ra = map[a], rb = map[b];
        if (kind[ra] != kind[rb]) return kind[ra] < kind[rb];
        if (ent[ra] != ent[rb]) return ent[ra] < ent[rb];
        return per[ra] < per[rb];
    });
    return o;
}

// Run three independent host tasks at once; an exception in any of them
// (out of host memory) is rethrown on the calling thread after all end.
template <typename F1, typename F2, typename F3>
static void parallel3(F1 &&f1, F2 &&f2, F3 &&f3) {
    std::exception_ptr e1, e2;
    std::thread t1([&] { try { f1(); } catch (...) { e1 = std::current_exception(); } });
    std::thread t2([&] { try { f2(); } catch (...) { e2 = std::current_exception(); } });
    std::exception_ptr e3;
    try { f3(); } catch (...) { e3 = std::current_exception(); }
    t1.join();
    t2.join();
    for (auto &e : {e1, e2, e3})
        if (e) std::rethrow_exception(e);
}

static std::shared_ptr<const PsData> device_view(const std::shared_ptr<const PsData> &src, bool reorder,
                                                 std::vector<int32_t> &prow, std::vector<int32_t> &pcol) {
    const PsData &p = *src;
    const int m = p.m(), n = p.n();
    prow.clear();
    pcol.clear();
    if (!reorder) {
        prow.resize(m); pcol.resize(n);
        for (int i = 0; i < m; i++) prow[i] = i;
        for (int j = 0; j < n; j++) pcol[j] = j;
        return src;
    }
    static const RawLp kNoLabels;
    const RawLp &R = p.raw ? *p.raw : kNoLabels;
    // the three orders are independent: equality rows, ">=" rows, columns (host threads)
    std::vector<int32_t> prow_ge;
    parallel3([&] { window_order(p.A.rowptr, entity_order(0, p.m_eq, p.row_map, R.row_kind, R.row_idx, R.row_t), prow); },
              [&] { window_order(p.A.rowptr, entity_order(p.m_eq, m, p.row_map, R.row_kind, R.row_idx, R.row_t), prow_ge); },
              [&] { window_order(p.AT.rowptr, entity_order(0, n, p.col_map, R.col_kind, R.col_idx, R.col_t), pcol); });
    prow.insert(prow.end(), prow_ge.begin(), prow_ge.end());
    // columns with more than kLongRow entries go last, in their order: the
    // primal kernel gives each of them a warp
    std::vector<int32_t> longc;
    {
        std::vector<int32_t> shortc;
        shortc.reserve(n);
        for (int32_t j : pcol) (p.AT.rowptr[j + 1] - p.AT.rowptr[j] > kLongRow ? longc : shortc).push_back(j);
        if (!longc.empty()) {
            pcol.swap(shortc);
            pcol.insert(pcol.end(), longc.begin(), longc.end());
        }
    }
    std::vector<int32_t> irow(m), icol(n);
    for (int i = 0; i < m; i++) irow[prow[i]] = i;
    for (int j = 0; j < n; j++) icol[pcol[j]] = j;
    auto d = std::make_shared<PsData>();
    d->raw = p.raw;
    d->m_eq = p.m_eq;
    d->value_bits = p.value_bits;
    d->eta = p.eta; d->omega0 = p.omega0; d->norm_A = p.norm_A; d->norm_bound = p.norm_bound; d->obj_const = p.obj_const;
    d->q_inf = p.q_inf; d->c_inf = p.c_inf;
    d->long_cols = (int)longc.size();
    auto permute_csr = [](const Csr &A, const std::vector<float> &v32, const std::vector<int32_t> &order,
                          const std::vector<int32_t> &inv_cols, Csr &out, std::vector<float> &o32) {
        out.rows = A.rows; out.cols = A.cols;
        out.rowptr.assign(1, 0);
        out.colidx.reserve(A.colidx.size()); out.val.reserve(A.val.size());
        if (!v32.empty()) o32.reserve(v32.size());
        for (int32_t r : order) {
            for (int32_t k = A.rowptr[r]; k < A.rowptr[r + 1]; k++) {
                out.colidx.push_back(inv_cols[A.colidx[k]]);
                out.val.push_back(A.val[k]);
                if (!v32.empty()) o32.push_back(v32[k]);
            }
            out.rowptr.push_back((int32_t)out.colidx.size());
        }
    };
    parallel3([&] { permute_csr(p.A, p.A_val32, prow, icol, d->A, d->A_val32); },
              [&] { permute_csr(p.AT, p.AT_val32, pcol, irow, d->AT, d->AT_val32); }, [] {});
    auto gather = [](const std::vector<double> &v, const std::vector<int32_t> &order) {
        std::vector<double> o(order.size());
        for (size_t t = 0; t < order.size(); t++) o[t] = v[order[t]];
        return o;
    };
    d->c = gather(p.c, pcol); d->l = gather(p.l, pcol); d->u = gather(p.u, pcol); d->Dc = gather(p.Dc, pcol);
    d->q = gather(p.q, prow); d->Dr = gather(p.Dr, prow);
    return d;
}

// same scaled matrix (structure, values as stored, equality rows)
static bool same_matrix(const PsData &a, const PsData &b) {
    return a.n() == b.n() && a.m() == b.m() && a.m_eq == b.m_eq && a.value_bits == b.value_bits &&
           a.A.rowptr == b.A.rowptr && a.A.colidx == b.A.colidx && a.A.val == b.A.val && a.A_val32 == b.A_val32;
}

// Period-strided groups of a device-order matrix.  In the entity-major layout
// consecutive rows are one constraint of one entity in consecutive periods,
// and the variables they use sit in consecutive device columns.  A group of
// kStrideRows consecutive rows is "strided" when all its rows have the same
// number of entries k and, for every entry q, row s of the group has column
// col_q + s and value val_q: the group is then described by k (column, value)
// slots instead of kStrideRows * k entries.  Other groups have k = -1.  Entry
// order within a row is kept, so a kernel summing the slots in order does the
// row's arithmetic in the same order as the CSR row.
constexpr int kStrideRows = 16;

struct StridedGroups {
    std::vector<int32_t> k;     // per group: entries per row, or -1
    std::vector<int32_t> off;   // per group: first slot (groups + 1 offsets)
    std::vector<int32_t> col;   // per slot: device column of the group's first row
    std::vector<double> val;    // per slot: the value all rows of the group share
};

static StridedGroups strided_groups(const Csr &M) {
    StridedGroups g;
    const int rows = M.rows;
    const int ng = (rows + kStrideRows - 1) / kStrideRows;
    g.k.assign(ng, -1);
    g.off.assign((size_t)ng + 1, 0);
    for (int gi = 0; gi < ng; gi++) {
        g.off[gi] = (int32_t)g.col.size();
        const int r0 = gi * kStrideRows;
        if (r0 + kStrideRows > rows) continue;   // a ragged last group stays on the CSR path
        const int k = M.rowptr[r0 + 1] - M.rowptr[r0];
        bool ok = k > 0;
        for (int s = 1; ok && s < kStrideRows; s++) {
            const int r = r0 + s;
            if (M.rowptr[r + 1] - M.rowptr[r] != k) { ok = false; break; }
            for (int q = 0; q < k; q++) {
                const int32_t e0 = M.rowptr[r0] + q, e = M.rowptr[r] + q;
                if (M.colidx[e] != M.colidx[e0] + s || M.val[e] != M.val[e0]) { ok = false; break; }
            }
        }
        if (!ok) continue;
        g.k[gi] = k;
        for (int q = 0; q < k; q++) {
            g.col.push_back(M.colidx[M.rowptr[r0] + q]);
            g.val.push_back(M.val[M.rowptr[r0] + q]);
        }
    }
    g.off[ng] = (int32_t)g.col.size();
    return g;
}

// Slot records of the period-strided groups of a stored CSR matrix (global
// indices, values as stored): sk[g] = k and the records of group g at
// 16 g + q when the group is strided with k <= 16 entries per row, else
// sk[g] = -1.  Values are compared bit for bit.  Record layout as SlotT:
// int32 column at byte 0, the value at byte 8 (FP64) or 4 (FP32).  The slot
// area must be zeroed.  Returns the rows in strided groups.
template <typename VT>
static int64_t build_slots(const int32_t *rp, const int32_t *ci, const VT *v, int64_t rows, signed char *sk,
                           char *sl) {
    const size_t rec = sizeof(VT) == 8 ? 16 : 8, voff = sizeof(VT) == 8 ? 8 : 4;
    const int64_t ng = (rows + kStrideRows - 1) / kStrideRows;
    int64_t covered = 0;
    for (int64_t g = 0; g < ng; g++) {
        sk[g] = -1;
        const int64_t r0 = g * kStrideRows;
        if (r0 + kStrideRows > rows) continue;
        const int k = rp[r0 + 1] - rp[r0];
        if (k <= 0 || k > kStrideRows) continue;
        bool ok = true;
        for (int s = 1; ok && s < kStrideRows; s++) {
            const int64_t r = r0 + s;
            if (rp[r + 1] - rp[r] != k) { ok = false; break; }
            for (int q = 0; q < k; q++) {
                const int64_t e0 = rp[r0] + q, e = rp[r] + q;
                if (ci[e] != ci[e0] + s || std::memcmp(v + e, v + e0, sizeof(VT)) != 0) { ok = false; break; }
            }
        }
        if (!ok) continue;
        sk[g] = (signed char)k;
        for (int q = 0; q < k; q++) {
            char *p = sl + (size_t)(r0 + q) * rec;
            std::memcpy(p, ci + rp[r0] + q, 4);
            std::memcpy(p + voff, v + rp[r0] + q, sizeof(VT));
        }
        covered += kStrideRows;
    }
    return covered;
}

// natural-order vector -> device order (and back)
static std::vector<double> to_device(const double *v, const std::vector<int32_t> &order) {
    std::vector<double> o(order.size());
    for (size_t t = 0; t < order.size(); t++) o[t] = v[order[t]];
    return o;
}
static void to_natural(std::vector<double> &v, const std::vector<int32_t> &order) {
    std::vector<double> o(v.size());
    for (size_t t = 0; t < order.size(); t++) o[order[t]] = v[t];
    v.swap(o);
}

static Scalars make_scalars(const uc_session &X, const PsData &p, double omega = 0.0) {
    Scalars s{};
    const double w = omega > 0.0 ? omega : p.omega0;
    s.eta = p.eta;
    s.omega = w;
    s.tau = p.eta / w;
    s.sigma = p.eta * w;
    s.tol = X.o.tol_rel_kkt;
    s.q_inf = p.q_inf;
    s.c_inf = p.c_inf;
    s.max_iter = X.o.max_iter;
    s.n_eval = X.o.n_eval;
    s.kkt_prev = INFINITY;
    s.status = NEEDS_INIT;
    s.algo = X.algo;
    s.metric = X.o.restart_metric;
    s.adaptive = X.adaptive ? 1 : 0;
    s.ad_eta = p.eta;
    s.ad_tau = p.eta / w;
    s.ad_sigma = p.eta * w;
    s.inv_next = 1.0 / (double)X.o.n_eval;
    s.pw_kp = X.o.pw_kp;
    s.pw_ki = X.o.pw_ki;
    s.pw_kd = X.o.pw_kd;
    s.pw_guard = X.o.pw_guard;
    s.stop_abs = X.polish_tol;
    return s;
}

// host twin of the device okey(): doubles in the same order as int64 keys
static long long order_key(double v) {
    long long b;
    std::memcpy(&b, &v, 8);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}

static void derived_vectors(const PsData &p, std::vector<double> &idc, std::vector<double> &idr,
                            std::vector<long long> &lk, std::vector<long long> &uk) {
    idc.resize(p.n()); idr.resize(p.m()); lk.resize(p.n()); uk.resize(p.n());
    for (int j = 0; j < p.n(); j++) {
        idc[j] = 1.0 / p.Dc[j];
        lk[j] = order_key(p.l[j]);
        uk[j] = order_key(p.u[j]);
    }
    for (int i = 0; i < p.m(); i++) idr[i] = 1.0 / p.Dr[i];
}

// start point, initial scalars and per-LP vectors of LP i into the staging image
static void stage_lp(uc_session &X, std::vector<char> &st, int i, const double *wx_nat, const double *wy_nat,
                     double womega) {
    const PsData &p = *X.Pd[i];
    std::vector<double> wxv, wyv;
    if (wx_nat) wxv = to_device(wx_nat, X.pcol[i]);
    if (wy_nat) wyv = to_device(wy_nat, X.prow[i]);
    const double *wx = wx_nat ? wxv.data() : nullptr;
    const double *wy = wy_nat ? wyv.data() : nullptr;
    const Layout &L = X.L;
    // 8-byte vector elements of LP i: contiguous from its offset, or every
    // K-th element from lane i in a lanes session
    auto putv = [&](size_t base, int64_t off, const void *src, int count) {
        if (X.K == 1) {
            if (count) std::memcpy(st.data() + base + off * 8, src, (size_t)count * 8);
            return;
        }
        for (int t = 0; t < count; t++)
            std::memcpy(st.data() + base + ((size_t)t * X.K + i) * 8, (const char *)src + (size_t)t * 8, 8);
    };
    putv(L.c, X.coff[i], p.c.data(), p.n());
    putv(L.l, X.coff[i], p.l.data(), p.n());
    putv(L.u, X.coff[i], p.u.data(), p.n());
    putv(L.Dc, X.coff[i], p.Dc.data(), p.n());
    putv(L.q, X.roff[i], p.q.data(), p.m());
    putv(L.Dr, X.roff[i], p.Dr.data(), p.m());
    {
        std::vector<double> idc, idr;
        std::vector<long long> lk, uk;
        derived_vectors(p, idc, idr, lk, uk);
        putv(L.inv_Dc, X.coff[i], idc.data(), p.n());
        putv(L.inv_Dr, X.roff[i], idr.data(), p.m());
        putv(L.lkey, X.coff[i], lk.data(), p.n());
        putv(L.ukey, X.coff[i], uk.data(), p.n());
    }
    std::vector<double> x0(p.n()), y0(p.m());
    for (int c = 0; c < p.n(); c++) x0[c] = std::min(std::max(wx ? wx[c] : 0.0, p.l[c]), p.u[c]);
    for (int r = 0; r < p.m(); r++) {
        const double v = wy ? wy[r] : 0.0;
        y0[r] = r >= p.m_eq ? std::max(v, 0.0) : v;
    }
    putv(L.x_init, X.coff[i], x0.data(), p.n());
    putv(L.y_init, X.roff[i], y0.data(), p.m());
    X.S_init[i] = make_scalars(X, p, womega);
    put(st, L.S_init + sizeof(Scalars) * i, &X.S_init[i], 1);
}

// evaluation, record reduction and controller (mode 0: start point, 1: regular)
static void launch_eval(uc_session &X, cudaStream_t s, int mode) {
    const dim3 grid(X.n_se, X.K);
    if (X.K == 1) {
        if (X.vb == 32) k_eval<float, 1><<<grid, kThreads, 0, s>>>(X.dse, X.b, mode);
        else k_eval<double, 1><<<grid, kThreads, 0, s>>>(X.dse, X.b, mode);
    } else if (X.K == 2) {
        if (X.vb == 32) k_eval<float, 2><<<grid, kThreads, 0, s>>>(X.dse, X.b, mode);
        else k_eval<double, 2><<<grid, kThreads, 0, s>>>(X.dse, X.b, mode);
    } else {
        if (X.vb == 32) k_eval<float, 4><<<grid, kThreads, 0, s>>>(X.dse, X.b, mode);
        else k_eval<double, 4><<<grid, kThreads, 0, s>>>(X.dse, X.b, mode);
    }
    k_reduce<<<X.k * kPart, kThreads, 0, s>>>(X.drg, X.b, mode);
    k_control<<<(32 * X.k + kControlThreads - 1) / kControlThreads, kControlThreads, 0, s>>>(X.b, mode, X.k);
}

// iteration kernels of the session's algorithm
// Launch an iteration kernel; with `pdl` it may overlap the tail of the
// iteration kernel before it (programmatic stream serialization).
template <typename Kern, typename... Args>
static cudaError_t launch_k(Kern kern, int grid, int block, cudaStream_t s, bool pdl, Args... args) {
    if (grid <= 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <typename VT, bool PRIMAL>
static cudaError_t launch_staged(const uc_session &X, cudaStream_t s, bool pdl, int it, int src) {
    const int grid = PRIMAL ? X.g_p : X.g_d;
    if (grid <= 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kStRows);
    cfg.dynamicSmemBytes = PRIMAL ? X.smem_p : X.smem_d;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k_iter_staged<VT, PRIMAL>, PRIMAL ? X.dcp : X.dcd, PRIMAL ? X.dgp : X.dgd,
                              X.b, it, src, X.stages);
}

template <typename VT, int ALGO, int BS, bool SD>
static cudaError_t launch_rows(const uc_session &X, cudaStream_t s, bool pdl, int it, int src, bool primal) {
    if (primal) {
        const int ns = (int)X.Nr - (X.k == 1 ? X.Pd[0]->long_cols : 0);
        const Uniform u = X.k == 1 ? Uniform{ns, 0, X.rpt[0], (ns + BS * X.rpt[0] - 1) / (BS * X.rpt[0]), (int)X.Nr}
                                   : Uniform{0, 0, 0, 0, 0};
        return launch_k(k_primal<VT, ALGO, BS, SD>, X.n_sp, BS, s, pdl, X.dsp, X.b, it, src, u);
    }
    const Uniform u = X.k == 1 ? Uniform{(int)X.Mr, X.m_eq[0], X.rpt[0], INT_MAX, (int)X.Mr} : Uniform{0, 0, 0, 0, 0};
    return launch_k(k_dual<VT, ALGO, BS, SD>, X.n_sd, BS, s, pdl, X.dsd, X.b, it, src, u);
}

template <int ALGO, int BS>
static void launch_iter(uc_session &X, cudaStream_t s, int it, int src, bool primal) {
    // the first primal kernel of a block follows the evaluation kernels: no overlap there
    const bool pdl = X.pdl && (!primal || it > 0);
    cudaError_t e;
    if (X.K > 1) {   // lanes session: 128-thread CTAs, K/2 threads per row
        const int grid = primal ? X.n_sp : X.n_sd;
        const Seg *segs = primal ? X.dsp : X.dsd;
        if (X.vb == 32) {
            if (X.K == 2) e = launch_k(primal ? k_primal_lanes<float, 2, 128> : k_dual_lanes<float, 2, 128>, grid, 128, s, pdl, segs, X.b, it, src);
            else e = launch_k(primal ? k_primal_lanes<float, 4, 128> : k_dual_lanes<float, 4, 128>, grid, 128, s, pdl, segs, X.b, it, src);
        } else {
            if (X.K == 2) e = launch_k(primal ? k_primal_lanes<double, 2, 128> : k_dual_lanes<double, 2, 128>, grid, 128, s, pdl, segs, X.b, it, src);
            else e = launch_k(primal ? k_primal_lanes<double, 4, 128> : k_dual_lanes<double, 4, 128>, grid, 128, s, pdl, segs, X.b, it, src);
        }
        if (e != cudaSuccess && X.launch_err == cudaSuccess) X.launch_err = e;
        return;
    }
    if (X.staged) {
        if (X.vb == 32) e = primal ? launch_staged<float, true>(X, s, pdl, it, src) : launch_staged<float, false>(X, s, pdl, it, src);
        else e = primal ? launch_staged<double, true>(X, s, pdl, it, src) : launch_staged<double, false>(X, s, pdl, it, src);
        if (e != cudaSuccess && X.launch_err == cudaSuccess) X.launch_err = e;
        return;
    }
    if (X.vb == 32) e = X.strided ? launch_rows<float, ALGO, BS, true>(X, s, pdl, it, src, primal)
                                  : launch_rows<float, ALGO, BS, false>(X, s, pdl, it, src, primal);
    else e = X.strided ? launch_rows<double, ALGO, BS, true>(X, s, pdl, it, src, primal)
                       : launch_rows<double, ALGO, BS, false>(X, s, pdl, it, src, primal);
    if (e != cudaSuccess && X.launch_err == cudaSuccess) X.launch_err = e;
}
template <int ALGO>
static void launch_iter_bs(uc_session &X, cudaStream_t s, int it, int src, bool primal) {
    switch (X.cta) {
        case 128: launch_iter<ALGO, 128>(X, s, it, src, primal); break;
        case 512: launch_iter<ALGO, 512>(X, s, it, src, primal); break;
        default: launch_iter<ALGO, 256>(X, s, it, src, primal); break;
    }
}
static void launch_primal(uc_session &X, cudaStream_t s, int it, int src) {
    if (X.algo == ALG_HALPERN) launch_iter_bs<ALG_HALPERN>(X, s, it, src, true);
    else launch_iter_bs<ALG_AVERAGE>(X, s, it, src, true);
}
static void launch_dual(uc_session &X, cudaStream_t s, int it, int src) {
    if (X.algo == ALG_HALPERN) launch_iter_bs<ALG_HALPERN>(X, s, it, src, false);
    else launch_iter_bs<ALG_AVERAGE>(X, s, it, src, false);
}
static void launch_apply(uc_session &X, cudaStream_t s) {
    if (!X.n_sa) return;
    if (X.K > 1) {   // lanes session: 128-thread segments, one grid row per lane
        const int ncol = (int)((X.Nr + 127) / 128);
        if (X.K == 2) k_apply<128, 2><<<dim3(X.n_sa, 2), 128, 0, s>>>(X.dsa, ncol, X.b);
        else k_apply<128, 4><<<dim3(X.n_sa, 4), 128, 0, s>>>(X.dsa, ncol, X.b);
        return;
    }
    switch (X.cta) {
        case 128: k_apply<128, 1><<<X.n_sa, 128, 0, s>>>(X.dsa, X.n_sac, X.b); break;
        case 512: k_apply<512, 1><<<X.n_sa, 512, 0, s>>>(X.dsa, X.n_sac, X.b); break;
        default: k_apply<256, 1><<<X.n_sa, 256, 0, s>>>(X.dsa, X.n_sac, X.b); break;
    }
}

// n_eval attempts of the adaptive step, then the move of the current iterate
// to buffer 0 (before the evaluation)
static void launch_adaptive(uc_session &X, cudaStream_t s, int it, const std::function<void(int)> &rec) {
    const int n = (int)X.Nr, m = (int)X.Mr;
    const int nbp = (n + kAdThreads - 1) / kAdThreads, nbd = (m + kAdThreads - 1) / kAdThreads;
    rec(0);
    if (nbp) {
        if (X.vb == 32) k_ad_primal<float><<<nbp, kAdThreads, 0, s>>>(X.b, n, it);
        else k_ad_primal<double><<<nbp, kAdThreads, 0, s>>>(X.b, n, it);
    }
    rec(1);
    if (nbd) {
        if (X.vb == 32) k_ad_dual<float><<<nbd, kAdThreads, 0, s>>>(X.b, m, X.m_eq[0], it, nbp);
        else k_ad_dual<double><<<nbd, kAdThreads, 0, s>>>(X.b, m, X.m_eq[0], it, nbp);
    }
    rec(2);
    k_ad_decide<<<1, 1024, 0, s>>>(X.b, nbp, nbd, it);
}
static void launch_adaptive_norm(uc_session &X, cudaStream_t s) {
    const int n = (int)X.Nr, m = (int)X.Mr;
    const int ne = (n + m + 255) / 256;
    if (ne) k_ad_norm<<<ne, 256, 0, s>>>(X.b, n, m);
    k_ad_src0<<<1, 1, 0, s>>>(X.b);
}

using BlockKernel = void (*)(BlockPlan, Bufs);
template <typename VT>
static BlockKernel block_kernel_vt(int threads, bool one, bool limit) {
    if (limit) return k_block<double, kSmallThreads, true, true>;
    if (threads <= kSmallThreads) return one ? k_block<VT, kSmallThreads, true> : k_block<VT, kSmallThreads, false>;
    if (threads <= kMidThreads) return one ? k_block<VT, kMidThreads, true> : k_block<VT, kMidThreads, false>;
    return one ? k_block<VT, kBigThreads, true> : k_block<VT, kBigThreads, false>;
}
static BlockKernel block_kernel(const uc_session &X, int threads) {
    return X.vb == 32 ? block_kernel_vt<float>(threads, X.k == 1, false)
                      : block_kernel_vt<double>(threads, X.k == 1, X.plan.polls != kBlockPolls);
}
static int block_head(const uc_session &X) {
    return (int)(sizeof(BlockLp) * X.k + sizeof(double2) * (X.k == 1 ? X.o.n_eval + 1 : 0));
}

// all n_eval iterations of a block (cooperative: the CTAs wait on one another,
// so all of them are resident)
static void launch_block(uc_session &X, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(X.blk_ctas);
    cfg.blockDim = dim3(X.blk_threads);
    cfg.dynamicSmemBytes = X.blk_smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, block_kernel(X, X.blk_threads), X.plan, X.b);
    if (e != cudaSuccess && X.launch_err == cudaSuccess) X.launch_err = e;
}

static int block_pack(uc_session &X, int count) {
    const int per = kSmallThreads / 32, grid = (count + per - 1) / per;
    if (X.vb == 32) k_block_pack<float><<<grid, kSmallThreads, 0, X.s>>>(X.plan.tiles, count, X.plan.image, X.b);
    else k_block_pack<double><<<grid, kSmallThreads, 0, X.s>>>(X.plan.tiles, count, X.plan.image, X.b);
    UC_CUDA(cudaGetLastError());
    return UC_OK;
}

static int capture(uc_session &X, int gi) {
    cudaStream_t s = X.s;
    const bool timing = X.o.kernel_timing != 0;
    const Bufs &b = X.b;
    UC_CUDA(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
    cudaError_t err = cudaSuccess;
    auto rec = [&](int e) {
        if (timing && err == cudaSuccess) err = cudaEventRecordWithFlags(X.tev[gi][e], s, cudaEventRecordExternal);
    };
    // the timed pair is a mid-block iteration: steady-state L2 contents, and
    // only the event nodes around it break the programmatic overlap
    const int timed_it = X.o.n_eval / 2;
    if (X.block) launch_block(X, s);
    if (X.block && timing && err == cudaSuccess)
        err = cudaMemcpyAsync(X.h_stamp + 2 * gi, X.plan.stamp, 2 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, s);
    for (int it = 0; !X.block && it < X.o.n_eval; it++) {
        if (X.adaptive) {
            launch_adaptive(X, s, it, [&](int e) { if (it == timed_it) rec(e); });
            continue;
        }
        const int src = it & 1;
        if (it == timed_it) rec(0);
        if (X.n_sp) launch_primal(X, s, it, src);
        if (it == timed_it) rec(1);
        if (X.n_sd) launch_dual(X, s, it, src);
        if (it == timed_it) rec(2);
    }
    if (X.adaptive) launch_adaptive_norm(X, s);
    launch_eval(X, s, 1);
    launch_apply(X, s);
    if (err == cudaSuccess) err = cudaGetLastError();
    if (err == cudaSuccess && X.launch_err != cudaSuccess) err = X.launch_err;
    if (err == cudaSuccess)
        err = cudaMemcpyAsync(X.h_status, b.status, sizeof(int) * X.k, cudaMemcpyDeviceToHost, s);
    cudaGraph_t g = nullptr;
    cudaError_t ce = cudaStreamEndCapture(s, &g);
    if (err != cudaSuccess) {
        if (g) cudaGraphDestroy(g);
        set_error("recording the iteration graph failed: %s", cudaGetErrorString(err));
        return UC_ECUDA;
    }
    if (ce != cudaSuccess) { set_error("graph capture failed: %s", cudaGetErrorString(ce)); return UC_ECUDA; }
    X.graph[gi] = g;
    UC_CUDA(cudaGraphInstantiate(&X.exec[gi], g, 0));
    return UC_OK;
}

// launches of one replay without a graph (use_graph = 0)
static int launch_direct(uc_session &X) {
    cudaStream_t s = X.s;
    const Bufs &b = X.b;
    if (X.block) launch_block(X, s);
    for (int it = 0; !X.block && it < X.o.n_eval; it++) {
        if (X.adaptive) {
            launch_adaptive(X, s, it, [](int) {});
            continue;
        }
        const int src = it & 1;
        if (X.n_sp) launch_primal(X, s, it, src);
        if (X.n_sd) launch_dual(X, s, it, src);
    }
    if (X.adaptive) launch_adaptive_norm(X, s);
    launch_eval(X, s, 1);
    launch_apply(X, s);
    UC_CUDA(cudaGetLastError());
    UC_CUDA(X.launch_err);
    UC_CUDA(cudaMemcpyAsync(X.h_status, b.status, sizeof(int) * X.k, cudaMemcpyDeviceToHost, s));
    return UC_OK;
}

// Shared memory and resident CTAs of the staged kernels for this session.
template <typename VT>
static int staged_setup_vt(uc_session &X) {
    X.smem_p = kStHead + X.stages * StLayout<VT, 5>::kBytes;
    X.smem_d = kStHead + X.stages * StLayout<VT, 3>::kBytes;
    int dev = 0, sms = 0, bp = 0, bd = 0;
    UC_CUDA(cudaGetDevice(&dev));
    UC_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // the attribute is per kernel, not per session: allow the largest stage count
    const int max_p = kStHead + kStMaxStages * StLayout<VT, 5>::kBytes;
    const int max_d = kStHead + kStMaxStages * StLayout<VT, 3>::kBytes;
    UC_CUDA(cudaFuncSetAttribute(k_iter_staged<VT, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_p));
    UC_CUDA(cudaFuncSetAttribute(k_iter_staged<VT, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_d));
    UC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bp, k_iter_staged<VT, true>, kStRows, X.smem_p));
    UC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bd, k_iter_staged<VT, false>, kStRows, X.smem_d));
    if (bp < 1 || bd < 1) {
        set_error("staged kernels: %d stages do not fit in shared memory", X.stages);
        return UC_EINVAL;
    }
    X.gmax_p = bp * sms;
    X.gmax_d = bd * sms;
    return UC_OK;
}
static int staged_setup(uc_session &X) {
    return X.vb == 32 ? staged_setup_vt<float>(X) : staged_setup_vt<double>(X);
}

// CTA tables of the LPs with mask[i]: every CTA works on a slice of one LP.
// LPs outside the mask get no CTAs (and an empty evaluation range).
static void build_tables(const uc_session &X, const std::vector<char> &mask, std::vector<Seg> &sp,
                         std::vector<Seg> &sd, std::vector<Seg> &se, std::vector<Seg> &sa,
                         std::vector<InstRange> &ranges, int &n_sac) {
    sp.clear(); sd.clear(); se.clear(); sa.clear();
    std::vector<Seg> sac;
    n_sac = 0;
    ranges.assign(X.k, InstRange{0, 0});
    if (X.K > 1) {
        // lanes session: one structure; K/2 threads per row in the iteration
        // kernels, one thread per element in the apply kernel (grid.y = lane)
        const int rows = X.cta / (X.K / 2);
        const int eq_end = X.m_eq[0];
        for (int64_t s = 0; s < X.Nr; s += rows) sp.push_back({0, (int)s, (int)std::min<int64_t>(s + rows, X.Nr), 0, 1});
        for (int64_t s = 0; s < X.Mr; s += rows) sd.push_back({0, (int)s, (int)std::min<int64_t>(s + rows, X.Mr), eq_end, 1});
        const int er = eval_rows(X.Mr + X.Nr);
        for (int64_t s = 0; s < X.Mr; s += er) se.push_back({0, (int)s, (int)std::min<int64_t>(s + er, X.Mr), eq_end << 1, 1});
        for (int64_t s = 0; s < X.Nr; s += er) se.push_back({0, (int)s, (int)std::min<int64_t>(s + er, X.Nr), 1, 1});
        if (se.empty()) se.push_back({0, 0, 0, 0, 1});
        for (int i = 0; i < X.k; i++) ranges[i] = {i * (int)se.size(), (i + 1) * (int)se.size()};
        for (int64_t s = 0; s < X.Nr; s += X.cta) sa.push_back({0, (int)s, (int)std::min<int64_t>(s + X.cta, X.Nr), 0, 1});
        n_sac = (int)sa.size();
        for (int64_t s = 0; s < X.Mr; s += X.cta) sa.push_back({0, (int)s, (int)std::min<int64_t>(s + X.cta, X.Mr), 0, 1});
        return;
    }
    for (int i = 0; i < X.k; i++) {
        if (!mask[i]) continue;
        const int64_t c0 = X.coff[i], c1 = X.coff[i + 1], r0 = X.roff[i], r1 = X.roff[i + 1];
        const int rpt = X.rpt[i];
        const int cta = X.cta * rpt;
        // the LP's long columns (last in its range) get one warp each (rpt = 0)
        const int64_t cl = c1 - X.Pd[i]->long_cols;
        for (int64_t s = c0; s < cl; s += cta) sp.push_back({i, (int)s, (int)std::min<int64_t>(s + cta, cl), 0, rpt});
        for (int64_t s = cl; s < c1; s += X.cta / 32) sp.push_back({i, (int)s, (int)std::min<int64_t>(s + X.cta / 32, c1), 0, 0});
        for (int64_t s = c0; s < c1; s += cta) sac.push_back({i, (int)s, (int)std::min<int64_t>(s + cta, c1), 0, rpt});
        const int eq_end = (int)(r0 + X.m_eq[i]);
        for (int64_t s = r0; s < r1; s += cta) sd.push_back({i, (int)s, (int)std::min<int64_t>(s + cta, r1), eq_end, rpt});
        ranges[i].eval_begin = (int)se.size();
        const int er = eval_rows(c1 - c0 + r1 - r0);
        for (int64_t s = r0; s < r1; s += er) se.push_back({i, (int)s, (int)std::min<int64_t>(s + er, r1), eq_end << 1, 1});
        for (int64_t s = c0; s < cl; s += er) se.push_back({i, (int)s, (int)std::min<int64_t>(s + er, cl), 1, 1});
        for (int64_t s = cl; s < c1; s += kThreads / 32) se.push_back({i, (int)s, (int)std::min<int64_t>(s + kThreads / 32, c1), 1, 0});
        if (se.size() == (size_t)ranges[i].eval_begin) se.push_back({i, 0, 0, 0, 1});
        ranges[i].eval_end = (int)se.size();
    }
    // the apply kernel covers columns and rows with one thread per element
    n_sac = (int)sac.size();
    sa = sac;
    sa.insert(sa.end(), sd.begin(), sd.end());
}

// bit r - a: row r of M, of rows [a, b), does not go on a run of the rows before it
// (see BlockTile); values as stored, v32: the FP32 values, if M is stored so
static unsigned tile_runs(const Csr &M, const std::vector<float> &v32, int a, int b) {
    unsigned runs = 1;
    for (int r = a + 1; r < b; r++) {
        const int p = M.rowptr[r - 1], e = M.rowptr[r], k = M.rowptr[r + 1] - e;
        bool same = e - p == k;
        for (int q = 0; same && q < k; q++)
            same = M.colidx[e + q] == M.colidx[p + q] + 1 &&
                   (v32.empty() ? M.val[e + q] == M.val[p + q] : v32[e + q] == v32[p + q]);
        if (!same) runs |= 1u << (r - a);
    }
    return runs;
}

static bool tile_before(const BlockTile &a, const BlockTile &b) {
    return a.kmax != b.kmax ? a.kmax > b.kmax : a.bytes > b.bytes;
}

// Tiles of LP i, primal and dual, the longest rows first, then the most bytes; cut once
// for a session, since an LP's matrix stays.
static void cut_tiles(uc_session &X, int i) {
    const PsData &v = *X.Pd[i];
    const int n = v.n(), m = v.m(), nl = v.long_cols, m_eq = X.m_eq[i];
    auto add = [&](int r0, unsigned info, int kmax, unsigned runs) {
        const int count = __builtin_popcount(runs);
        X.cut[i][tile_primal(info)].push_back(BlockTile{r0, info, kmax, runs, 0, 0, tile_bytes(tile_stride(kmax, count), count), 0});
    };
    auto cut = [&](const Csr &M, int a, int b, int64_t base, bool primal, bool ineq) {
        for (int s = a; s < b; s += kTileRows) {
            const int e = std::min(b, s + kTileRows);
            int kmax = 0, kmin = INT_MAX;
            for (int r = s; r < e; r++) {
                kmax = std::max(kmax, M.rowptr[r + 1] - M.rowptr[r]);
                kmin = std::min(kmin, M.rowptr[r + 1] - M.rowptr[r]);
            }
            const unsigned runs = tile_runs(M, primal ? v.AT_val32 : v.A_val32, s, e);
            const int kind = kmin == kmax && kmax >= 1 && kmax <= kUniform ? TILE_UNIFORM : TILE_ANY;
            add((int)(base + s), tile_info(e - s, kind, primal, ineq, i), kmax, runs);
        }
    };
    cut(v.AT, 0, n - nl, X.coff[i], true, false);
    for (int j = n - nl; j < n; j++)
        add((int)(X.coff[i] + j), tile_info(1, TILE_LONG, true, false, i), (v.AT.rowptr[j + 1] - v.AT.rowptr[j] + 31) / 32, ~0u);
    cut(v.A, 0, m_eq, X.roff[i], false, false);
    cut(v.A, m_eq, m, X.roff[i], false, true);
    for (auto &t : X.cut[i]) std::stable_sort(t.begin(), t.end(), tile_before);
}

// Tiles of the resident block kernel for the LPs in `mask`, dealt to the warps of
// at most one CTA per SM: primal tiles, longest rows first, to the warps in turn
// over the CTAs, dual tiles in turn from the last warp back, so that a warp has
// tiles of one phase while there are warps enough and the longest rows get a warp
// of their own.  Sets X.block: the tiles fit into the CTAs' shared memory.
static void plan_block(uc_session &X, const std::vector<char> &mask, std::vector<BlockTile> &tiles,
                       std::vector<BlockWarp> &warps) {
    tiles.clear();
    warps.clear();
    X.block = false;
    if (!X.block_able) return;
    X.cut.resize(X.k);
    std::vector<BlockTile> t[2];   // dual, primal
    int64_t bytes = 0;
    for (int i = 0; i < X.k; i++) {
        if (!mask[i]) continue;
        if (X.cut[i][0].empty() && X.cut[i][1].empty()) cut_tiles(X, i);
        for (const auto &list : X.cut[i]) for (const BlockTile &T : list) bytes += T.bytes;
        if (bytes > (int64_t)X.sms * X.blk_smem_max) return;
    }
    for (int ph = 0; ph < 2; ph++) {   // the LPs' lists merged, equal tiles in the LPs' order
        std::vector<size_t> ends{0};
        for (int i = 0; i < X.k; i++)
            if (mask[i]) {
                t[ph].insert(t[ph].end(), X.cut[i][ph].begin(), X.cut[i][ph].end());
                ends.push_back(t[ph].size());
            }
        for (size_t step = 1; step + 1 < ends.size(); step *= 2)
            for (size_t a = 0; a + step + 1 < ends.size(); a += 2 * step)
                std::inplace_merge(t[ph].begin() + ends[a], t[ph].begin() + ends[a + step],
                                   t[ph].begin() + ends[std::min(a + 2 * step, ends.size() - 1)], tile_before);
    }
    const int64_t np = t[1].size(), nd = t[0].size();
    if (np == 0 || nd == 0) return;
    const int nc = (int)std::min<int64_t>(X.sms, std::max(np, nd));
    const bool big = np + nd > (int64_t)kBigTiles * nc * (kMidThreads / 32);
    const int W = (int)std::min<int64_t>((big ? kBigThreads : kMidThreads) / 32, (np + nd + nc - 1) / nc);
    const int64_t S = (int64_t)nc * W;
    const int head = block_head(X);
    int64_t most = 0, image = 0;
    tiles.reserve((size_t)(np + nd));
    warps.reserve((size_t)S);
    for (int c = 0; c < nc; c++) {
        int64_t at = head + (big ? W * kStageBytes : 0);
        for (int w = 0; w < W; w++) {
            const int64_t slot = (int64_t)w * nc + c;
            const size_t first = tiles.size();
            for (int ph = 1; ph >= 0; ph--)
                for (int64_t q = ph ? slot : S - 1 - slot; q < (ph ? np : nd); q += S) {
                    BlockTile T = t[ph][q];
                    T.smem = (int)at;
                    T.img = (int)(image / 16);
                    at += T.bytes;
                    image += T.bytes - kTileOwn;
                    tiles.push_back(T);
                }
            warps.push_back(BlockWarp{(int)first, (int)(tiles.size() - first)});
        }
        most = std::max(most, at);
    }
    if (most > X.blk_smem_max) return;
    X.blk_image = image;
    X.plan.head = head;
    X.plan.nlps = X.k;
    X.plan.n_eval = X.o.n_eval;
    X.blk_ctas = nc;
    X.blk_threads = 32 * W;
    X.blk_smem = (int)most;
    X.block = true;
}

// Chunk lists of the staged kernels for the LPs in `mask`: rows are cut into
// chunks of at most kStRows rows and kStEnts entries, in device order; the
// chunks are then dealt to at most `gmax` CTAs by longest-processing-time
// first on their streamed bytes (so CTAs finish together), and each CTA's
// chunks are kept in row order.  `ctas` gets the CTA ranges (size CTAs + 1).
static void build_chunks(const uc_session &X, const std::vector<char> &mask, bool primal, int gmax,
                         std::vector<Chunk> &out, std::vector<int> &ctas) {
    std::vector<Chunk> all;
    std::vector<double> cost;
    const double per_row = primal ? 5 * 8 + 4 : 3 * 8 + 4, per_ent = 4 + (double)X.vs + 8;
    for (int i = 0; i < X.k; i++) {
        if (!mask[i]) continue;
        const Csr &M = primal ? X.Pd[i]->AT : X.Pd[i]->A;
        const int64_t base = primal ? X.coff[i] : X.roff[i], zo = X.zoff[i];
        const int rows = M.rows;
        const int aux = primal ? 0 : (int)(X.roff[i] + X.m_eq[i]);
        for (int r = 0; r < rows;) {
            int r1 = std::min(rows, r + kStRows);
            while (M.rowptr[r1] - M.rowptr[r] > kStEnts) r1--;   // rows are no longer than kStEnts
            all.push_back({i, (int)(base + r), (int)(base + r1), (int)(zo + M.rowptr[r]), (int)(zo + M.rowptr[r1]), aux});
            cost.push_back(per_row * (r1 - r) + per_ent * (M.rowptr[r1] - M.rowptr[r]));
            r = r1;
        }
    }
    const int g = std::max(1, std::min<int>(gmax, (int)all.size()));
    std::vector<int> order(all.size());
    for (size_t t = 0; t < order.size(); t++) order[t] = (int)t;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return cost[a] > cost[b]; });
    using Load = std::pair<double, int>;
    std::priority_queue<Load, std::vector<Load>, std::greater<Load>> heap;
    for (int c = 0; c < g; c++) heap.push({0.0, c});
    std::vector<std::vector<int>> bins(g);
    for (int t : order) {
        Load l = heap.top();
        heap.pop();
        bins[l.second].push_back(t);
        heap.push({l.first + cost[t], l.second});
    }
    out.clear();
    ctas.assign(1, 0);
    for (auto &bin : bins) {
        std::sort(bin.begin(), bin.end());
        for (int t : bin) out.push_back(all[t]);
        ctas.push_back((int)out.size());
    }
}

static int capture(uc_session &X, int gi);

// Rebuild the tables for the LPs in `mask` and re-capture the graphs; the
// stream must be idle.  Used when LPs finish (compaction) or are reset.
static int retable(uc_session &X, const std::vector<char> &mask) {
    std::vector<Seg> sp, sd, se, sa;
    std::vector<InstRange> ranges;
    build_tables(X, mask, sp, sd, se, sa, ranges, X.n_sac);
    const Layout &L = X.L;
    auto up = [&](size_t off, const void *src, size_t bytes) -> int {
        if (bytes) UC_CUDA(cudaMemcpyAsync(X.D + off, src, bytes, cudaMemcpyHostToDevice, X.s));
        return UC_OK;
    };
    int rc = up(L.segs_p, sp.data(), sizeof(Seg) * sp.size());
    if (!rc) rc = up(L.segs_d, sd.data(), sizeof(Seg) * sd.size());
    if (!rc) rc = up(L.segs_e, se.data(), sizeof(Seg) * se.size());
    if (!rc) rc = up(L.segs_a, sa.data(), sizeof(Seg) * sa.size());
    if (!rc) rc = up(L.ranges, ranges.data(), sizeof(InstRange) * ranges.size());
    std::vector<BlockTile> tiles;
    std::vector<BlockWarp> warps;
    plan_block(X, mask, tiles, warps);
    if (!rc && X.block) rc = up(L.tiles, tiles.data(), sizeof(BlockTile) * tiles.size());
    if (!rc && X.block) rc = up(L.warps, warps.data(), sizeof(BlockWarp) * warps.size());
    if (!rc && X.block) rc = block_pack(X, (int)tiles.size());
    std::vector<Chunk> cp, cd;
    std::vector<int> gp, gd;
    if (X.staged) {
        build_chunks(X, mask, true, X.gmax_p, cp, gp);
        build_chunks(X, mask, false, X.gmax_d, cd, gd);
        if (!rc) rc = up(L.chunks_p, cp.data(), sizeof(Chunk) * cp.size());
        if (!rc) rc = up(L.chunks_d, cd.data(), sizeof(Chunk) * cd.size());
        if (!rc) rc = up(L.ctas_p, gp.data(), sizeof(int) * gp.size());
        if (!rc) rc = up(L.ctas_d, gd.data(), sizeof(int) * gd.size());
    }
    if (rc) return rc;
    if (X.staged) {
        // no chunks at all (no LP tabled) leaves one empty CTA
        X.g_p = cp.empty() ? 0 : (int)gp.size() - 1;
        X.g_d = cd.empty() ? 0 : (int)gd.size() - 1;
    }
    X.n_sp = (int)sp.size(); X.n_sd = (int)sd.size(); X.n_se = (int)se.size(); X.n_sa = (int)sa.size();
    X.tabled = mask;
    X.retables++;
    UC_CUDA(cudaStreamSynchronize(X.s));
    if (X.o.use_graph) {
        for (int gi = 0; gi < 2; gi++) {
            if (X.exec[gi]) { cudaGraphExecDestroy(X.exec[gi]); X.exec[gi] = nullptr; }
            if (X.graph[gi]) { cudaGraphDestroy(X.graph[gi]); X.graph[gi] = nullptr; }
        }
        for (int gi = 0; gi < (X.o.kernel_timing ? 2 : 1); gi++) {
            int r2 = capture(X, gi);
            if (r2) return r2;
        }
    }
    return UC_OK;
}

static bool live_status(int st) { return st == RUNNING || st == NEEDS_INIT; }

// resident: the session may take memory for the resident kernel, a lanes session then
// storing its LPs one after another (see below); set to whether it did
static int session_create_as(const PsData *const *Pp, const std::shared_ptr<const PsData> *owners, int k,
                             const uc_solve_opts &o, cudaStream_t user_stream, bool &resident, uc_session **out) {
    *out = nullptr;
    const bool may = resident;
    resident = false;
    if (k < 1) { set_error("need at least one LP"); return UC_EINVAL; }
    if (o.n_eval < 2 || (o.n_eval & 1)) { set_error("n_eval must be even and >= 2"); return UC_EINVAL; }
    if (o.max_iter < 0) { set_error("max_iter must be >= 0"); return UC_EINVAL; }
    auto *X = new (std::nothrow) uc_session();
    if (!X) { set_error("out of host memory"); return UC_ENOMEM; }
    std::unique_ptr<uc_session> guard(X);
    X->k = k;
    X->o = o;
    X->vb = Pp[0]->value_bits;
    if (o.spmv_kernel < 0 || o.spmv_kernel > 2) { set_error("spmv_kernel must be 0, 1 or 2"); return UC_EINVAL; }
    if (o.stages != 0 && (o.stages < 2 || o.stages > kStMaxStages)) {
        set_error("stages must be 0 or 2..%d", kStMaxStages);
        return UC_EINVAL;
    }
    if (o.algorithm < 0 || o.algorithm > 1 || o.restart_metric < 0 || o.restart_metric > 2) {
        set_error("algorithm must be 0 or 1 and restart_metric 0, 1 or 2");
        return UC_EINVAL;
    }
    X->algo = o.algorithm;
    if (o.polish != 0 && o.polish != 1) { set_error("polish must be 0 or 1"); return UC_EINVAL; }
    if (o.polish && (o.algorithm != ALG_HALPERN || o.lanes || o.adaptive_step || !(o.tol_abs_feas > 0.0) ||
                     o.polish_max_iter < 0)) {
        set_error("polish needs the Halpern algorithm, no lanes, tol_abs_feas > 0 and polish_max_iter >= 0");
        return UC_EINVAL;
    }
    if (!(std::isfinite(o.pw_kp) && std::isfinite(o.pw_ki) && std::isfinite(o.pw_kd)) || o.pw_kp < 0 ||
        o.pw_ki < 0 || o.pw_kd < 0) {
        set_error("pw_kp, pw_ki and pw_kd must be finite and >= 0");
        return UC_EINVAL;
    }
    if (!std::isfinite(o.pw_guard) || o.pw_guard < 0 || (o.pw_guard > 0 && o.pw_guard < 1)) {
        set_error("pw_guard must be 0 (off) or a finite value >= 1");
        return UC_EINVAL;
    }
    if (o.adaptive_step != 0 && o.adaptive_step != 1) { set_error("adaptive_step must be 0 or 1"); return UC_EINVAL; }
    X->adaptive = o.adaptive_step == 1;
    if (X->adaptive && (X->algo != ALG_AVERAGE || k != 1 || o.lanes || o.spmv_kernel == 2)) {
        set_error("adaptive_step needs algorithm 1 (iterate averaging), one LP, no lanes, row kernels");
        return UC_EINVAL;
    }
    if (o.cta_rows != 0 && o.cta_rows != 128 && o.cta_rows != 256 && o.cta_rows != 512) {
        set_error("cta_rows must be 0, 128, 256 or 512");
        return UC_EINVAL;
    }
    X->cta = o.cta_rows ? o.cta_rows : 128;
    X->pdl = o.no_pdl == 0;
    X->vs = X->vb == 32 ? 4 : 8;
    X->P.assign(owners, owners + k);
    X->reorder = o.no_reorder == 0;
    X->Pd.resize(k); X->prow.resize(k); X->pcol.resize(k);
    for (int i = 0; i < k; i++) X->Pd[i] = device_view(X->P[i], X->reorder, X->prow[i], X->pcol[i]);
    for (int i = 1; i < k; i++)
        if (Pp[i]->value_bits != X->vb) { set_error("batched LPs must share value_bits"); return UC_EINVAL; }
    if (X->vb == 32)   // the kernels widen FP32 values by moving bits: normal, nonzero values only
        for (int i = 0; i < k; i++)
            for (float f : Pp[i]->A_val32)
                if (!std::isnormal(f)) { set_error("FP32 matrix value %g is zero, subnormal or not finite", (double)f); return UC_EINVAL; }
    if (o.lanes) {
        if (k != 2 && k != 4) { set_error("lanes sessions hold 2 or 4 LPs (got %d)", k); return UC_EINVAL; }
        if (X->algo != ALG_HALPERN || o.spmv_kernel == 2) {
            set_error("lanes sessions run the Halpern algorithm on the row kernels");
            return UC_EINVAL;
        }
        for (int i = 1; i < k; i++)
            if (!same_matrix(*X->Pd[i], *X->Pd[0])) {
                set_error("lanes sessions need LPs with one scaled matrix (LP %d differs from LP 0)", i);
                return UC_EINVAL;
            }
    }
    // offsets of the LPs; interleaved: one structure, every LP starts at row, column and entry 0
    auto lay_out = [&](bool interleaved) {
        X->K = interleaved ? k : 1;
        X->roff.assign(k + 1, 0); X->coff.assign(k + 1, 0); X->zoff.assign(k + 1, 0);
        if (interleaved) {
            X->M = (int64_t)Pp[0]->m() * k; X->N = (int64_t)Pp[0]->n() * k; X->Z = Pp[0]->A.nnz();
            X->Mr = Pp[0]->m(); X->Nr = Pp[0]->n();
            X->roff[k] = X->Mr; X->coff[k] = X->Nr; X->zoff[k] = X->Z;
        } else {
            for (int i = 0; i < k; i++) {
                X->roff[i + 1] = X->roff[i] + Pp[i]->m();
                X->coff[i + 1] = X->coff[i] + Pp[i]->n();
                X->zoff[i + 1] = X->zoff[i] + Pp[i]->A.nnz();
            }
            X->M = X->roff[k]; X->N = X->coff[k]; X->Z = X->zoff[k];
            X->Mr = X->M; X->Nr = X->N;
        }
        // row indices are also stored shifted left by one bit in the evaluation table
        return X->M < (1LL << 30) && X->N < INT32_MAX && X->Z < INT32_MAX;
    };
    if (!lay_out(o.lanes && !may) && (!o.lanes || !lay_out(true))) {
        set_error("batch too large for int32 indices");
        return UC_EINVAL;
    }

    X->rpt.assign(k, 1);
    X->m_eq.assign(k, 0);
    for (int i = 0; i < k; i++) {
        const int r = (o.rows_per_thread && o.rows_per_thread[i]) ? o.rows_per_thread[i] : 1;
        if (r != 1 && r != 2 && r != 4) { set_error("rows_per_thread must be 1, 2 or 4"); return UC_EINVAL; }
        X->rpt[i] = r;
        X->m_eq[i] = Pp[i]->m_eq;
    }
    // staged kernels (spmv_kernel 2; measured slower than the row kernels on
    // the 6,049-bus LP, so opt-in): Halpern only, every matrix row within one chunk
    X->staged = o.spmv_kernel == 2;
    X->stages = o.stages ? o.stages : 2;
    if (X->staged) {
        int longest = 0;
        for (int i = 0; i < k; i++)
            for (const Csr *M : {&X->Pd[i]->A, &X->Pd[i]->AT})
                for (int r = 0; r < M->rows; r++) longest = std::max(longest, M->rowptr[r + 1] - M->rowptr[r]);
        if (X->algo != ALG_HALPERN || longest > kStEnts) {
            set_error("staged kernels need the Halpern algorithm and rows of at most %d entries (longest %d)",
                      kStEnts, longest);
            return UC_EINVAL;
        }
        int rc = staged_setup(*X);
        if (rc) return rc;
    }
    // resident block kernel: Halpern row sessions
    std::vector<BlockTile> tiles;
    std::vector<BlockWarp> warps;
    {
        int dev = 0, coop = 0;
        UC_CUDA(cudaGetDevice(&dev));
        UC_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
        UC_CUDA(cudaDeviceGetAttribute(&X->sms, cudaDevAttrMultiProcessorCount, dev));
        UC_CUDA(cudaDeviceGetAttribute(&X->blk_smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
        X->blk_smem_max -= 1024;   // the kernel's static part
        X->block_able = may && coop && o.spmv_kernel == 0 && X->algo == ALG_HALPERN && X->K == 1 && k <= kBlockMaxLps &&
                        o.n_eval <= kBlockMaxEval;
        if (X->block_able)
            for (int nt : {kSmallThreads, kMidThreads, kBigThreads})
                UC_CUDA(cudaFuncSetAttribute(block_kernel(*X, nt), cudaFuncAttributeMaxDynamicSharedMemorySize, X->blk_smem_max));
        plan_block(*X, std::vector<char>(k, 1), tiles, warps);
        if (k == 1 && !X->block) X->block_able = false;   // no subset of its LPs fits either
    }
    // A lanes session whose LPs fit into shared memory one after another runs the
    // resident kernel: two LPs of 474 k rows and columns 14.3 us per iteration (the
    // interleaved kernels 18.0), four of 95 k 6.9 (13.0).  Its tables hold all LPs to its
    // end, and the matrix is stored once per LP.  Else the vectors are interleaved.
    if (o.lanes && !X->block) {
        lay_out(true);
        X->block_able = false;
        X->cta = 128;   // the lanes kernels are built for 128-thread CTAs
    }
    resident = X->block_able;
    if (!X->block_able) X->cut.clear();
    const int64_t M = X->M, N = X->N, Z = X->Z;
    // CTA tables for every LP (their sizes are the capacities of the device tables)
    std::vector<Seg> sp, sd, se, sa;
    std::vector<InstRange> ranges;
    std::vector<char> all(k, 1);
    build_tables(*X, all, sp, sd, se, sa, ranges, X->n_sac);
    X->tabled = all;
    std::vector<Chunk> cp, cd;
    std::vector<int> gp, gd;
    if (X->staged) {
        build_chunks(*X, all, true, X->gmax_p, cp, gp);
        build_chunks(*X, all, false, X->gmax_d, cd, gd);
        X->cap_cp = (int)cp.size(); X->cap_cd = (int)cd.size();
        X->g_p = cp.empty() ? 0 : (int)gp.size() - 1;
        X->g_d = cd.empty() ? 0 : (int)gd.size() - 1;
    }
    X->n_sp = X->cap_sp = (int)sp.size(); X->n_sd = X->cap_sd = (int)sd.size();
    X->n_se = X->cap_se = (int)se.size(); X->n_sa = X->cap_sa = (int)sa.size();

    Layout &L = X->L;
    size_t off = 0;
    // 16 bytes of slack after every array: the staged kernels' copies round
    // their windows out to 16-byte boundaries
    auto take = [&](size_t n) { size_t p = off; off += align_up(std::max<size_t>(n, 1) + 16, 256); return p; };
    const size_t vs = X->vs;
    // +4 zero entries: a 16-byte load starting inside the array stays inside it
    const int64_t Mr = X->Mr, Nr = X->Nr;   // rows of A and A^T as stored
    L.A_rp = take((Mr + 1) * 4); L.A_ci = take((Z + 4) * 4); L.A_v = take((Z + 4) * vs);
    L.AT_rp = take((Nr + 1) * 4); L.AT_ci = take((Z + 4) * 4); L.AT_v = take((Z + 4) * vs);
    X->strided = o.spmv_kernel == 0 && X->K == 1 && !X->staged;
    const int64_t gA = X->strided ? (Mr + kStrideRows - 1) / kStrideRows : 0;
    const int64_t gAT = X->strided ? (Nr + kStrideRows - 1) / kStrideRows : 0;
    const size_t slot_bytes = X->vb == 32 ? sizeof(SlotT<float>) : sizeof(SlotT<double>);
    L.A_sk = take(gA); L.AT_sk = take(gAT);
    L.A_sl = take(gA * kStrideRows * slot_bytes); L.AT_sl = take(gAT * kStrideRows * slot_bytes);
    L.segs_p = take(sizeof(Seg) * X->n_sp); L.segs_d = take(sizeof(Seg) * X->n_sd);
    L.segs_e = take(sizeof(Seg) * X->n_se); L.segs_a = take(sizeof(Seg) * X->n_sa);
    L.ranges = take(sizeof(InstRange) * k);
    L.chunks_p = take(sizeof(Chunk) * X->cap_cp); L.chunks_d = take(sizeof(Chunk) * X->cap_cd);
    L.ctas_p = take(sizeof(int) * (X->gmax_p + 1)); L.ctas_d = take(sizeof(int) * (X->gmax_d + 1));
    const int nW = (int)std::min<long long>((long long)o.max_iter + 1, 1LL << 22);
    L.W = take(sizeof(double) * nW); L.W1 = take(sizeof(double) * nW);
    const int64_t nAd = X->adaptive ? (int64_t)o.max_iter : 0;
    L.adS = take(sizeof(double) * nAd); L.adG = take(sizeof(double) * nAd);
    L.c = take(N * 8); L.l = take(N * 8); L.u = take(N * 8); L.Dc = take(N * 8);
    L.inv_Dc = take(N * 8); L.lkey = take(N * 8); L.ukey = take(N * 8);
    L.q = take(M * 8); L.Dr = take(M * 8); L.inv_Dr = take(M * 8);
    L.x_init = take(N * 8); L.y_init = take(M * 8); L.S_init = take(sizeof(Scalars) * k);
    {   // tables for any subset of the LPs: a tile per 32 rows or columns begun (rows: of either kind), or per long column
        int64_t nt = 0;
        for (int i = 0; i < k && X->block_able; i++) {
            const PsData &p = *X->Pd[i];
            nt += (p.n() + kTileRows - 1) / kTileRows + (p.m() + kTileRows - 1) / kTileRows + 1 + p.long_cols;
        }
        L.tiles = take(sizeof(BlockTile) * nt);
        L.warps = take(X->block_able ? sizeof(BlockWarp) * 32 * X->sms : 0);
    }
    L.upload_end = off;
    // packed on the device: the image of all LPs; that of a subset in the CTAs' shared memory where all do not fit
    L.image = take(X->block ? X->blk_image : X->block_able ? (size_t)X->sms * X->blk_smem_max : 0);
    L.x0 = take(N * 8); L.x1 = take(N * 8); L.y0 = take(M * 8); L.y1 = take(M * 8);
    L.xsum = take(N * 8); L.ysum = take(M * 8); L.xa = take(N * 8); L.ya = take(M * 8);
    L.xret = take(N * 8); L.yret = take(M * 8);
    L.xt = take(X->block_able ? N * 16 : 0);
    L.yt = take(X->block_able ? M * 16 : 0);
    L.blk_seq = take(sizeof(unsigned));
    L.stamp = take(2 * sizeof(unsigned long long));
    L.part = take(sizeof(double) * kPart * X->n_se * X->K);
    L.adp = take(X->adaptive ? sizeof(double) * (size_t)((Nr + kAdThreads - 1) / kAdThreads + 2 * ((Mr + kAdThreads - 1) / kAdThreads)) : 0);
    L.lane_stage = take(X->K > 1 ? (size_t)4 * (Nr + Mr) * 8 : 0);
    L.red = take(sizeof(double) * kPart * k);
    L.S = take(sizeof(Scalars) * k);
    L.status = take(sizeof(int) * k);
    L.total = off;

    auto t0 = std::chrono::steady_clock::now();
    std::vector<char> st(L.upload_end);
    X->S_init.resize(k);
    {
        int32_t *arp = (int32_t *)(st.data() + L.A_rp), *atrp = (int32_t *)(st.data() + L.AT_rp);
        int32_t *aci = (int32_t *)(st.data() + L.A_ci), *atci = (int32_t *)(st.data() + L.AT_ci);
        for (int i = 0; i < k; i++) {
            const PsData &p = *X->Pd[i];
            const int64_t ro = X->roff[i], co = X->coff[i], zo = X->zoff[i];
            if (X->K > 1 && i > 0) {   // lanes session: the matrix is stored once
                stage_lp(*X, st, i, nullptr, nullptr, 0.0);
                continue;
            }
            for (int r = 0; r < p.m(); r++) arp[ro + r] = (int32_t)(p.A.rowptr[r] + zo);
            for (int c = 0; c < p.n(); c++) atrp[co + c] = (int32_t)(p.AT.rowptr[c] + zo);
            for (int64_t z = 0; z < p.A.nnz(); z++) {
                aci[zo + z] = (int32_t)(p.A.colidx[z] + co);
                atci[zo + z] = (int32_t)(p.AT.colidx[z] + ro);
            }
            if (X->vb == 32) {
                put(st, L.A_v + zo * 4, p.A_val32.data(), p.A.nnz());
                put(st, L.AT_v + zo * 4, p.AT_val32.data(), p.A.nnz());
            } else {
                put(st, L.A_v + zo * 8, p.A.val.data(), p.A.nnz());
                put(st, L.AT_v + zo * 8, p.AT.val.data(), p.A.nnz());
            }
            stage_lp(*X, st, i, (k == 1) ? o.warm_x : nullptr, (k == 1) ? o.warm_y : nullptr,
                     (k == 1) ? o.warm_omega : 0.0);
        }
        arp[Mr] = (int32_t)Z;
        atrp[Nr] = (int32_t)Z;
        if (X->strided) {
            auto slots = [&](const int32_t *rp, const int32_t *ci, size_t v_off, int64_t rows, size_t sk_off,
                             size_t sl_off) {
                signed char *sk = (signed char *)(st.data() + sk_off);
                char *sl = st.data() + sl_off;
                return X->vb == 32 ? build_slots(rp, ci, (const float *)(st.data() + v_off), rows, sk, sl)
                                   : build_slots(rp, ci, (const double *)(st.data() + v_off), rows, sk, sl);
            };
            X->strided_rows_A = slots(arp, aci, L.A_v, Mr, L.A_sk, L.A_sl);
            X->strided_rows_AT = slots(atrp, atci, L.AT_v, Nr, L.AT_sk, L.AT_sl);
        }
        put(st, L.segs_p, sp.data(), X->n_sp);
        put(st, L.segs_d, sd.data(), X->n_sd);
        put(st, L.segs_e, se.data(), X->n_se);
        put(st, L.segs_a, sa.data(), X->n_sa);
        put(st, L.ranges, ranges.data(), k);
        if (X->block) {
            put(st, L.tiles, tiles.data(), tiles.size());
            put(st, L.warps, warps.data(), warps.size());
        }
        put(st, L.chunks_p, cp.data(), cp.size()); put(st, L.chunks_d, cd.data(), cd.size());
        put(st, L.ctas_p, gp.data(), gp.size()); put(st, L.ctas_d, gd.data(), gd.size());
        // Halpern weights, computed as the oracle's Halpern step computes them: w = (j+1)/(j+2), 1 - w
        double *W = (double *)(st.data() + L.W), *W1 = (double *)(st.data() + L.W1);
        for (int jj = 0; jj < nW; jj++) {
            W[jj] = ((double)jj + 1.0) / ((double)jj + 2.0);
            W1[jj] = 1.0 - W[jj];
        }
        // adaptive step factors of attempt a (k = a + 1 attempts, base k + 1 = a + 2),
        // with the host's pow as the oracle computes them
        double *adS = (double *)(st.data() + L.adS), *adG = (double *)(st.data() + L.adG);
        for (int64_t a = 0; a < nAd; a++) {
            adS[a] = 1.0 - std::pow((double)(a + 2), -0.3);
            adG[a] = 1.0 + std::pow((double)(a + 2), -0.6);
        }
    }

    if (user_stream) X->s = user_stream;
    else {
        UC_CUDA(cudaStreamCreateWithFlags(&X->s, cudaStreamNonBlocking));
        X->own_stream = true;
    }
    cudaStream_t s = X->s;
    X->bytes = L.total;
    if (o.alloc) {
        X->D = (char *)o.alloc(L.total, (void *)s, o.alloc_ctx);
        if (!X->D) { set_error("device allocator returned NULL for %zu bytes", L.total); return UC_ENOMEM; }
    } else {
        cudaError_t e = cudaMallocAsync((void **)&X->D, L.total, s);
        if (e != cudaSuccess) {
            X->D = nullptr;
            set_error("cudaMallocAsync(%zu) failed: %s", L.total, cudaGetErrorString(e));
            return e == cudaErrorMemoryAllocation ? UC_ENOMEM : UC_ECUDA;
        }
    }
    char *D = X->D;
    if ((uintptr_t)D & 255) { set_error("device allocation is not 256-byte aligned"); return UC_EINVAL; }
    UC_CUDA(cudaMemcpyAsync(D, st.data(), L.upload_end, cudaMemcpyHostToDevice, s));
    X->h2d = (long long)L.upload_end;
    Bufs &b = X->b;
    b.A_rp = (const int *)(D + L.A_rp); b.A_ci = (const int *)(D + L.A_ci); b.A_v = D + L.A_v;
    b.A_sk = (const signed char *)(D + L.A_sk); b.AT_sk = (const signed char *)(D + L.AT_sk);
    b.A_sl = D + L.A_sl; b.AT_sl = D + L.AT_sl;
    b.AT_rp = (const int *)(D + L.AT_rp); b.AT_ci = (const int *)(D + L.AT_ci); b.AT_v = D + L.AT_v;
    b.c = (const double *)(D + L.c); b.l = (const double *)(D + L.l); b.u = (const double *)(D + L.u);
    b.q = (const double *)(D + L.q); b.Dr = (const double *)(D + L.Dr); b.Dc = (const double *)(D + L.Dc);
    b.inv_Dr = (const double *)(D + L.inv_Dr); b.inv_Dc = (const double *)(D + L.inv_Dc);
    b.lkey = (const long long *)(D + L.lkey); b.ukey = (const long long *)(D + L.ukey);
    b.W = (const double *)(D + L.W); b.W1 = (const double *)(D + L.W1); b.nW = nW;
    b.adS = (const double *)(D + L.adS); b.adG = (const double *)(D + L.adG);
    b.adp = (double *)(D + L.adp);
    b.red = (double *)(D + L.red);
    b.x[0] = (double *)(D + L.x0); b.x[1] = (double *)(D + L.x1);
    b.y[0] = (double *)(D + L.y0); b.y[1] = (double *)(D + L.y1);
    b.xsum = (double *)(D + L.xsum); b.ysum = (double *)(D + L.ysum);
    b.xa = (double *)(D + L.xa); b.ya = (double *)(D + L.ya);
    b.xret = (double *)(D + L.xret); b.yret = (double *)(D + L.yret);
    b.part = (double *)(D + L.part);
    b.blk_seq = (unsigned *)(D + L.blk_seq);
    b.n_eval = o.n_eval;
    X->plan.tiles = (const BlockTile *)(D + L.tiles);
    X->plan.warps = (const BlockWarp *)(D + L.warps);
    X->plan.image = (unsigned char *)(D + L.image);
    X->plan.seq = b.blk_seq;
    X->plan.xt = (ulonglong2 *)(D + L.xt);
    X->plan.yt = (ulonglong2 *)(D + L.yt);
    X->plan.stamp = o.kernel_timing ? (unsigned long long *)(D + L.stamp) : nullptr;
    X->plan.stamp_it = o.n_eval / 2 - 1;   // its end is the next iteration's start
    b.S = (Scalars *)(D + L.S);
    b.status = (int *)(D + L.status);
    X->dsp = (const Seg *)(D + L.segs_p); X->dsd = (const Seg *)(D + L.segs_d);
    X->dse = (const Seg *)(D + L.segs_e); X->dsa = (const Seg *)(D + L.segs_a);
    X->drg = (const InstRange *)(D + L.ranges);
    X->dcp = (const Chunk *)(D + L.chunks_p); X->dcd = (const Chunk *)(D + L.chunks_d);
    X->dgp = (const int *)(D + L.ctas_p); X->dgd = (const int *)(D + L.ctas_d);
    // nothing runs until the first reset: mark every LP finished-as-idle
    UC_CUDA(cudaMemsetAsync(D + L.S, 0xff, sizeof(Scalars) * k, s));   // status -1: idle
    UC_CUDA(cudaMemsetAsync(D + L.status, 0xff, sizeof(int) * k, s));
    UC_CUDA(cudaMemsetAsync(D + L.blk_seq, 0, sizeof(unsigned), s));
    if (X->block) {
        int rc = block_pack(*X, (int)tiles.size());
        if (rc) return rc;
    }
    if (X->block_able) {   // tag 0: no iteration's
        UC_CUDA(cudaMemsetAsync(D + L.xt, 0, N * 16, s));
        UC_CUDA(cudaMemsetAsync(D + L.yt, 0, M * 16, s));
    }
    UC_CUDA(cudaMemsetAsync(D + L.stamp, 0, 2 * sizeof(unsigned long long), s));
    UC_CUDA(cudaHostAlloc((void **)&X->h_status, sizeof(int) * k, cudaHostAllocDefault));
    for (int i = 0; i < k; i++) X->h_status[i] = -1;
    X->active.assign(k, 0);
    const bool timing = o.kernel_timing != 0;
    for (auto &e : X->ev) UC_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    if (X->block_able && timing) {
        UC_CUDA(cudaHostAlloc((void **)&X->h_stamp, 4 * sizeof(unsigned long long), cudaHostAllocDefault));
        std::memset(X->h_stamp, 0, 4 * sizeof(unsigned long long));
    }
    if (o.use_graph) {
        for (int gi = 0; gi < 2; gi++) {
            if (timing)
                for (auto &e : X->tev[gi]) UC_CUDA(cudaEventCreate(&e));
            int rc = capture(*X, gi);
            if (rc) return rc;
            if (!timing) break;   // one graph suffices without per-replay events
        }
    }
    UC_CUDA(cudaStreamSynchronize(s));
    X->upload_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    *out = guard.release();
    return UC_OK;
}

// lanes sessions: LP `lane`'s elements of an interleaved vector <-> contiguous
// `count` elements at `host` (through the session's staging area, stream-ordered)
static int lane_upload(uc_session &X, double *dev_vec, int lane, const void *host, int count) {
    if (!count) return UC_OK;
    double *stage = (double *)(X.D + X.L.lane_stage);
    UC_CUDA(cudaMemcpyAsync(stage, host, (size_t)count * 8, cudaMemcpyHostToDevice, X.s));
    k_lane_copy<<<(count + 255) / 256, 256, 0, X.s>>>(dev_vec, stage, count, X.K, lane, 0);
    UC_CUDA(cudaGetLastError());
    return UC_OK;
}
static int lane_download(uc_session &X, void *host, const double *dev_vec, int lane, int count, size_t stage_off) {
    if (!count) return UC_OK;
    if (stage_off + (size_t)count > (size_t)4 * (X.Nr + X.Mr)) {
        set_error("lanes staging area too small");
        return UC_ECUDA;
    }
    double *stage = (double *)(X.D + X.L.lane_stage) + stage_off;
    k_lane_copy<<<(count + 255) / 256, 256, 0, X.s>>>(stage, dev_vec, count, X.K, lane, 1);
    UC_CUDA(cudaGetLastError());
    UC_CUDA(cudaMemcpyAsync(host, stage, (size_t)count * 8, cudaMemcpyDeviceToHost, X.s));
    return UC_OK;
}

// state of LP i (or all, i < 0) <- its start point; then the anchor KKT on the device
static int session_reset(uc_session &X, int which) {
    cudaStream_t s = X.s;
    char *D = X.D;
    const Layout &L = X.L;
    const int i0 = which < 0 ? 0 : which, i1 = which < 0 ? X.k : which + 1;
    if (which >= X.k) { set_error("LP index %d out of range", which); return UC_EINVAL; }
    for (int i = i0; i < i1; i++) {
        const size_t cx = X.coff[i] * 8, nx = (X.coff[i + 1] - X.coff[i]) * 8;
        const size_t cy = X.roff[i] * 8, ny = (X.roff[i + 1] - X.roff[i]) * 8;
        if (X.K > 1) {
            const int n = (int)X.Nr, m = (int)X.Mr;
            if (n + m > 0)
                k_lane_reset<<<(n + m + 255) / 256, 256, 0, s>>>(X.b, (const double *)(D + L.x_init),
                                                                 (const double *)(D + L.y_init), n, m, X.K, i);
            UC_CUDA(cudaGetLastError());
        } else if (nx) {
            for (size_t dst : {L.x0, L.x1, L.xa, L.xret})
                UC_CUDA(cudaMemcpyAsync(D + dst + cx, D + L.x_init + cx, nx, cudaMemcpyDeviceToDevice, s));
            UC_CUDA(cudaMemsetAsync(D + L.xsum + cx, 0, nx, s));
        }
        if (X.K == 1 && ny) {
            for (size_t dst : {L.y0, L.y1, L.ya, L.yret})
                UC_CUDA(cudaMemcpyAsync(D + dst + cy, D + L.y_init + cy, ny, cudaMemcpyDeviceToDevice, s));
            UC_CUDA(cudaMemsetAsync(D + L.ysum + cy, 0, ny, s));
        }
        UC_CUDA(cudaMemcpyAsync(D + L.S + sizeof(Scalars) * i, D + L.S_init + sizeof(Scalars) * i,
                                sizeof(Scalars), cudaMemcpyDeviceToDevice, s));
        X.active[i] = 1;
        X.h_status[i] = NEEDS_INIT;
    }
    // the tables must hold every LP that is still iterating or about to start
    std::vector<char> want(X.k, 0);
    bool differ = false;
    for (int i = 0; i < X.k; i++) {
        want[i] = X.active[i] && live_status(X.h_status[i]);
        differ |= want[i] && !X.tabled[i];
    }
    if (differ) {
        int rc = retable(X, want);
        if (rc) return rc;
    }
    launch_eval(X, s, 0);
    X.launches += 3;
    UC_CUDA(cudaGetLastError());
    return UC_OK;
}

static bool all_done(const uc_session &X) {
    for (int i = 0; i < X.k; i++) {
        if (!X.active[i]) continue;
        const int st = ((volatile int *)X.h_status)[i];
        if (st == RUNNING || st == NEEDS_INIT) return false;
    }
    return true;
}

// replays until every active LP has stopped, or max_replays, cancel or timeout
static int session_run(uc_session &X, int max_replays) {
    cudaStream_t s = X.s;
    const bool timing = X.o.kernel_timing != 0 && X.o.use_graph;
    const int depth = 2;
    int launched = 0, checked = 0;
    X.host_status = UC_OK;
    auto t0 = std::chrono::steady_clock::now();
    while (true) {
        while (launched < max_replays && launched - checked < depth) {
            if (X.o.use_graph) UC_CUDA(cudaGraphLaunch(X.exec[timing ? (launched & 1) : 0], s));
            else { int rc = launch_direct(X); if (rc) return rc; }
            UC_CUDA(cudaEventRecord(X.ev[launched & 3], s));
            launched++;
            X.polls++;
            X.launches += X.block ? 5 : X.adaptive ? 3LL * X.o.n_eval + 6 : 2LL * X.o.n_eval + 4;
        }
        if (checked >= launched) break;
        UC_CUDA(cudaEventSynchronize(X.ev[checked & 3]));
        const int gi = checked & 1;
        checked++;
        const bool done = all_done(X);
        if (!done && X.o.use_graph) {
            int live = 0, tab = 0;
            std::vector<char> want(X.k, 0);
            for (int i = 0; i < X.k; i++) {
                want[i] = X.active[i] && live_status(((volatile int *)X.h_status)[i]);
                live += want[i];
                tab += X.tabled[i];
            }
            if (!X.o.lanes && live > 0 && 4 * live <= 3 * tab) {   // lanes sessions keep one table
                // drain the replay still in flight, then rebuild for the live LPs only
                UC_CUDA(cudaStreamSynchronize(s));
                checked = launched;
                for (int i = 0; i < X.k; i++) want[i] = X.active[i] && live_status(((volatile int *)X.h_status)[i]);
                if (!all_done(X)) {
                    int rc = retable(X, want);
                    if (rc) return rc;
                }
            }
        }
        if (timing && !done && X.block) {
            // the halves of an iteration overlap: its time is split by their FP64 instructions
            const volatile unsigned long long *t = X.h_stamp + 2 * gi;
            // a block that ends before the timed iteration leaves an older block's (cleared by
            // the kernel they cost 0.3 % of an iteration at 300 buses)
            if (t[0] != X.last_stamp && t[1] > t[0]) {
                X.last_stamp = t[0];
                const double ms = (double)(t[1] - t[0]) * 1e-6, p = (double)(X.Z + 4 * X.N), d = (double)(X.Z + 4 * X.M);
                X.tp_sum += ms * p / (p + d); X.td_sum += ms * d / (p + d); X.timed++;
            }
        } else if (timing && !done) {
            float a = 0.f, c = 0.f;
            if (cudaEventElapsedTime(&a, X.tev[gi][0], X.tev[gi][1]) == cudaSuccess &&
                cudaEventElapsedTime(&c, X.tev[gi][1], X.tev[gi][2]) == cudaSuccess) {
                X.tp_sum += a; X.td_sum += c; X.timed++;
            }
        }
        if (done) break;
        if (X.o.cancel && *X.o.cancel) { X.host_status = UC_ECANCELLED; break; }
        if (X.o.timeout_ms > 0) {
            const double ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
            if (ms > X.o.timeout_ms) { X.host_status = UC_ETIMEOUT; break; }
        }
    }
    UC_CUDA(cudaStreamSynchronize(s));
    UC_CUDA(cudaGetLastError());
    X.last_run_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    return UC_OK;
}

static int session_result(uc_session &X, int i, uc_result **out) {
    *out = nullptr;
    if (i < 0 || i >= X.k) { set_error("LP index %d out of range", i); return UC_EINVAL; }
    cudaStream_t s = X.s;
    Scalars S;
    UC_CUDA(cudaMemcpyAsync(&S, X.b.S + i, sizeof(Scalars), cudaMemcpyDeviceToHost, s));
    UC_CUDA(cudaStreamSynchronize(s));
    const PsData &p = *X.P[i];
    const int n = p.n(), m = p.m();
    auto *res = new (std::nothrow) uc_result();
    if (!res) { set_error("out of host memory"); return UC_ENOMEM; }
    std::unique_ptr<uc_result> guard(res);
    res->ps = X.P[i];
    const int n_eval = X.o.n_eval;
    const int part = X.o.max_iter % n_eval;
    // current iterate: buffer 0 after a full block; after a limit reached
    // inside a block, buffer (max_iter mod n_eval) & 1
    // (adaptive step: buffer 0 always, moved there before every evaluation)
    const int cur = (S.status == ITER_LIMIT && !X.adaptive) ? (part & 1) : 0;
    int j_now = S.j_base;
    if (S.status == ITER_LIMIT && part) j_now = S.j_base + part;
    res->x_cur.resize(n); res->y_cur.resize(m); res->x_avg.resize(n); res->y_avg.resize(m);
    const size_t cx = X.coff[i], cy = X.roff[i];
    // LP i's elements of a device vector (contiguous, or lane i of a lanes
    // session through its staging area: up to seven vectors, 3 n + 4 m doubles,
    // within its 4 (n + m))
    size_t stage_off = 0;
    auto d2h = [&](std::vector<double> &dst, const double *base, size_t off, int count) -> int {
        if (X.K == 1) {
            if (count) UC_CUDA(cudaMemcpyAsync(dst.data(), base + off, (size_t)count * 8, cudaMemcpyDeviceToHost, s));
            return UC_OK;
        }
        int rc = lane_download(X, dst.data(), base, i, count, stage_off);
        stage_off += (size_t)count;
        return rc;
    };
    int rc = d2h(res->x_cur, X.b.x[cur], cx, n);
    if (!rc) rc = d2h(res->y_cur, X.b.y[cur], cy, m);
    const bool halp = X.algo == ALG_HALPERN;
    // Halpern: "average" slot = epoch anchor; returned point = last map output
    if (!rc) rc = d2h(res->x_avg, halp ? X.b.xa : X.b.xsum, cx, n);
    if (!rc) rc = d2h(res->y_avg, halp ? X.b.ya : X.b.ysum, cy, m);
    if (!rc && (S.status == OPTIMAL || halp)) {
        res->x_ret.resize(n); res->y_ret.resize(m);
        rc = d2h(res->x_ret, X.b.xret, cx, n);
        if (!rc) rc = d2h(res->y_ret, X.b.yret, cy, m);
    }
    // infeasible: the Farkas direction y_hat - y_in (y_in = buffer 1 at a block end)
    std::vector<double> y_in;
    if (!rc && S.status == INFEASIBLE) {
        y_in.resize(m);
        rc = d2h(y_in, X.b.y[1], cy, m);
    }
    if (rc) return rc;
    UC_CUDA(cudaStreamSynchronize(s));
    if (S.status == INFEASIBLE) {
        res->y_ray.resize(m);
        for (int r = 0; r < m; r++) res->y_ray[r] = res->y_ret[r] - y_in[r];
        if (X.reorder) to_natural(res->y_ray, X.prow[i]);
    }
    if (!halp && X.adaptive) {   // step-weighted average (the current point before any accepted step)
        for (int c = 0; c < n; c++) res->x_avg[c] = S.wsum > 0.0 ? res->x_avg[c] / S.wsum : res->x_cur[c];
        for (int r = 0; r < m; r++) res->y_avg[r] = S.wsum > 0.0 ? res->y_avg[r] / S.wsum : res->y_cur[r];
        if (S.status != OPTIMAL) { res->x_ret = res->x_cur; res->y_ret = res->y_cur; }
    } else if (!halp) {
        for (int c = 0; c < n; c++) res->x_avg[c] = j_now ? res->x_avg[c] / j_now : res->x_cur[c];
        for (int r = 0; r < m; r++) res->y_avg[r] = j_now ? res->y_avg[r] / j_now : res->y_cur[r];
        if (S.status != OPTIMAL) { res->x_ret = res->x_cur; res->y_ret = res->y_cur; }
    }
    if (X.reorder) {   // device order -> the LP's own order
        for (auto *v : {&res->x_cur, &res->x_avg, &res->x_ret}) to_natural(*v, X.pcol[i]);
        for (auto *v : {&res->y_cur, &res->y_avg, &res->y_ret}) to_natural(*v, X.prow[i]);
    }
    uc_stats &o = res->stats;
    int status;
    if (S.status == OPTIMAL) status = UC_OK;
    else if (S.status == ITER_LIMIT) status = UC_EITERLIMIT;
    else if (S.status == NUMERIC) status = UC_ENUMERIC;
    else if (S.status == INFEASIBLE) status = UC_EINFEASIBLE;
    else if (S.status == STALLED) {
        status = UC_ECUDA;
        set_error(X.staged ? "a staged iteration kernel stopped waiting for its shared-memory copies"
                           : "the resident block kernel stopped waiting for another CTA's element");
    }
    else status = X.host_status ? X.host_status : UC_EITERLIMIT;
    o.status = status;
    o.iters = (S.status == ITER_LIMIT) ? X.o.max_iter : S.k_base;
    o.restarts = S.restarts;
    o.evals = S.evals;
    o.returned_average = (S.status == OPTIMAL && S.which == 1) ? 1 : 0;
    o.rel_primal = S.rel_p; o.rel_dual = S.rel_d; o.rel_gap = S.rel_g;
    o.abs_primal = S.abs_p;
    o.dual_objective = S.dobj + p.obj_const;
    o.omega = S.omega;
    o.solve_ms = X.last_run_ms;
    o.upload_ms = X.upload_ms;
    o.primal_kernel_ms = X.timed ? X.tp_sum / X.timed : 0.0;
    o.dual_kernel_ms = X.timed ? X.td_sum / X.timed : 0.0;
    o.timed_launches = X.timed;
    o.kernel_launches = (int)std::min<long long>(X.launches, INT32_MAX);
    o.rejected_steps = X.adaptive ? std::max(0, o.iters - S.ad_acc) : 0;
    o.h2d_bytes = X.h2d;
    o.d2h_bytes = (long long)(n + m) * 8 * ((S.status == OPTIMAL || halp) ? 3 : 2) + (long long)sizeof(Scalars) +
                  X.polls * 4LL * X.k;
    X.active[i] = 0;
    *out = guard.release();
    return status;
}

static int session_create(const PsData *const *Pp, const std::shared_ptr<const PsData> *owners, int k,
                          const uc_solve_opts &o, cudaStream_t user_stream, uc_session **out) {
    bool resident = true;
    int rc = session_create_as(Pp, owners, k, o, user_stream, resident, out);
    // the row kernels need 16 bytes per row and column and the image less (9 MB of 78 at
    // 391 k rows and columns), the interleaved layout holds the matrix once
    if (rc == UC_ENOMEM && resident) {
        resident = false;
        rc = session_create_as(Pp, owners, k, o, user_stream, resident, out);
    }
    return rc;
}

// fn(t, T) for t < T, on host threads where there is work for them; fn allocates and
// throws nothing
template <typename F>
static void in_chunks(int64_t total, F &&fn) {
    const int T = (int)std::max<int64_t>(1, std::min<int64_t>({8, (int64_t)std::thread::hardware_concurrency(), total >> 16}));
    std::vector<std::thread> th;
    int t = 1;
    try {
        th.reserve(T);
        for (; t < T; t++) th.emplace_back([&fn, t, T] { fn(t, T); });
    } catch (const std::exception &) {   // no thread to be had: here
        for (; t < T; t++) fn(t, T);
    }
    fn(0, T);
    for (auto &x : th) x.join();
}

// The slot's matrix stays, and with it the device order: the new LP's matrix is
// compared, and its vectors are put into that order and their derived ones computed,
// by up to eight host threads in one pass, into pinned memory that the session keeps
// (64 bytes per column and 32 per row of its largest LP; pageable memory if there is
// none).  0.8 ms at 474 k rows and columns; building a new device view for it, of
// which the order and the permuted matrix are most, took 20.5.
static int session_update_lp(uc_session &X, int i, const std::shared_ptr<const PsData> &np) {
    if (i < 0 || i >= X.k) { set_error("LP index %d out of range", i); return UC_EINVAL; }
    const PsData &a = *X.P[i], &p = *np;
    const int n = a.n(), m = a.m();
    std::atomic<bool> same{n == p.n() && m == p.m() && a.m_eq == p.m_eq && a.value_bits == p.value_bits &&
                           a.A.rowptr.size() == p.A.rowptr.size() && a.A.colidx.size() == p.A.colidx.size() &&
                           a.A.val.size() == p.A.val.size()};
    std::vector<double> plain;
    double *st = nullptr;
    if (same) {
        if (!X.h_vec) {
            int64_t most = 0;
            for (int q = 0; q < X.k; q++) most = std::max<int64_t>(most, 8 * (int64_t)X.P[q]->n() + 4 * (int64_t)X.P[q]->m());
            if (cudaMallocHost((void **)&X.h_vec, (size_t)std::max<int64_t>(1, most) * 8) != cudaSuccess) {
                cudaGetLastError();
                X.h_vec = nullptr;
            }
        }
        if (!X.h_vec) plain.resize((size_t)8 * n + (size_t)4 * m);
        st = X.h_vec ? X.h_vec : plain.data();
        const int64_t nz = (int64_t)a.A.colidx.size();
        const int32_t *pc = X.pcol[i].data(), *pr = X.prow[i].data();
        const size_t N = n, M = m;
        double *row = st + 8 * N;
        in_chunks(nz + n + m, [&](int t, int T) {
            auto part = [&](int64_t len, int64_t &b, int64_t &e) { b = len * t / T; e = len * (t + 1) / T; };
            int64_t b, e;
            part((int64_t)a.A.rowptr.size(), b, e);
            if (!std::equal(a.A.rowptr.begin() + b, a.A.rowptr.begin() + e, p.A.rowptr.begin() + b)) same = false;
            part(nz, b, e);
            if (!std::equal(a.A.colidx.begin() + b, a.A.colidx.begin() + e, p.A.colidx.begin() + b) ||
                !std::equal(a.A.val.begin() + b, a.A.val.begin() + e, p.A.val.begin() + b)) same = false;
            part(n, b, e);
            for (int64_t j = b; j < e; j++) {
                const int32_t s = pc[j];
                const double l = p.l[s], u = p.u[s], d = p.Dc[s];
                const long long lk = order_key(l), uk = order_key(u);
                st[j] = p.c[s];
                st[N + j] = l;
                st[2 * N + j] = u;
                st[3 * N + j] = d;
                st[4 * N + j] = std::min(std::max(0.0, l), u);
                st[5 * N + j] = 1.0 / d;
                std::memcpy(st + 6 * N + j, &lk, 8);
                std::memcpy(st + 7 * N + j, &uk, 8);
            }
            part(m, b, e);
            for (int64_t r = b; r < e; r++) {
                const int32_t s = pr[r];
                row[r] = p.q[s];
                row[M + r] = p.Dr[s];
                row[2 * M + r] = 0.0;
                row[3 * M + r] = 1.0 / p.Dr[s];
            }
        });
    }
    if (!same) {
        set_error("update_lp: the new LP must have the same scaled matrix as slot %d", i);
        return UC_EINVAL;
    }
    X.P[i] = np;
    const Layout &L = X.L;
    auto upload = [&](size_t base, int64_t off, const double *v, int count) -> int {
        if (X.K > 1) return lane_upload(X, (double *)(X.D + base), i, v, count);
        if (count) UC_CUDA(cudaMemcpyAsync(X.D + base + off * 8, v, (size_t)count * 8, cudaMemcpyHostToDevice, X.s));
        return UC_OK;
    };
    int rc = 0, q = 0;
    for (size_t base : {L.c, L.l, L.u, L.Dc, L.x_init, L.inv_Dc, L.lkey, L.ukey})
        rc |= upload(base, X.coff[i], st + (size_t)n * q++, n);
    q = 0;
    for (size_t base : {L.q, L.Dr, L.y_init, L.inv_Dr}) rc |= upload(base, X.roff[i], st + (size_t)8 * n + (size_t)m * q++, m);
    if (rc) {
        cudaStreamSynchronize(X.s);
        set_error("update_lp: host-to-device copy failed");
        return UC_ECUDA;
    }
    X.S_init[i] = make_scalars(X, p);
    UC_CUDA(cudaMemcpyAsync(X.D + L.S_init + sizeof(Scalars) * i, &X.S_init[i], sizeof(Scalars),
                            cudaMemcpyHostToDevice, X.s));
    X.h2d += (8LL * n + 4LL * m) * 8 + (long long)sizeof(Scalars);
    UC_CUDA(cudaStreamSynchronize(X.s));
    return UC_OK;
}

static int session_set_start(uc_session &X, int i, const double *x, const double *y, double omega) {
    if (i < 0 || i >= X.k) { set_error("LP index %d out of range", i); return UC_EINVAL; }
    const PsData &p = *X.P[i];
    std::vector<double> xs(p.n()), ys(p.m());
    for (int c = 0; c < p.n(); c++) {
        const int32_t s = X.pcol[i][c];
        xs[c] = std::min(std::max(x ? x[s] : 0.0, p.l[s]), p.u[s]);
    }
    for (int r = 0; r < p.m(); r++) {
        const double v = y ? y[X.prow[i][r]] : 0.0;
        ys[r] = r >= p.m_eq ? std::max(v, 0.0) : v;
    }
    if (X.K > 1) {
        int rc = lane_upload(X, (double *)(X.D + X.L.x_init), i, xs.data(), p.n());
        if (!rc) rc = lane_upload(X, (double *)(X.D + X.L.y_init), i, ys.data(), p.m());
        if (rc) return rc;
    } else {
        if (p.n()) UC_CUDA(cudaMemcpyAsync(X.D + X.L.x_init + X.coff[i] * 8, xs.data(), p.n() * 8, cudaMemcpyHostToDevice, X.s));
        if (p.m()) UC_CUDA(cudaMemcpyAsync(X.D + X.L.y_init + X.roff[i] * 8, ys.data(), p.m() * 8, cudaMemcpyHostToDevice, X.s));
    }
    X.S_init[i] = make_scalars(X, p, omega);
    UC_CUDA(cudaMemcpyAsync(X.D + X.L.S_init + sizeof(Scalars) * i, &X.S_init[i], sizeof(Scalars),
                            cudaMemcpyHostToDevice, X.s));
    X.h2d += (long long)(p.n() + p.m()) * 8 + (long long)sizeof(Scalars);
    UC_CUDA(cudaStreamSynchronize(X.s));
    return UC_OK;
}

static int max_replays(const uc_session &X) { return X.o.max_iter / X.o.n_eval + 1; }

// ---------------------------------------------------------------------------
// KKT evaluation that allocates nothing (uc_kkt_noalloc)
//
// Some callers may not allocate device memory at all: processes whose device
// memory is reserved up front by their own pool allocator (a fresh driver
// allocation would then fail or fragment the pool), and latency-bound loops
// that must not enter the allocator, since cudaMalloc and cudaFree may
// synchronise the device.  For them this variant of the evaluation keeps its
// per-CTA partial sums in the file-scope array below instead of session memory.  Every GPU that loads
// this library holds the array (kNoAllocMaxBlocks * kNoAllocSlots doubles,
// 512 KiB) until the process exits.
// ---------------------------------------------------------------------------
constexpr int kNoAllocSlots = 8;         // Slot entries RP2 .. BND (DY2 stays 0)
constexpr int kNoAllocMaxBlocks = 8192;  // CTA records in the scratch
// Rows or columns per CTA: 256 (one per thread) while all CTAs are resident at
// once (four per SM), else 512 so, else 1024, which spreads a CTA's sums and its
// division over four rows per thread.  Measured: 47 k rows + columns 14.6 us at
// 256 (15.4 at 512), 227 k 20.9 us at 512 (27.4 at 256), 1.9 M 87.6 us at 1024
// (96.2 at 512).  The size limit is that of 1024: n/1024 + m/1024 <= 8192.
constexpr int kNoAllocRows = 1024;
constexpr int kNoAllocSmall = 256;
constexpr int kNoAllocCtas = 4;          // per SM (64 registers; 3 and 5 measured 5-7 % slower)
constexpr int kNoAllocGroup = 64;        // CTAs whose records the last of them to end adds up
constexpr int kNoAllocTickets = 16;      // counter sets, taken in turn by the calls

static __device__ __align__(256) double g_kkt_scratch[kNoAllocMaxBlocks * kNoAllocSlots];
// CTAs ended per group and groups ended; every counter wraps to zero with its
// last arrival.  A set per call in turn: calls that overlap against the contract
// spoil their own results (the scratch) but not the counts of later calls.
static __device__ unsigned g_kkt_ended[kNoAllocTickets][kNoAllocMaxBlocks / kNoAllocGroup + 1];

// row . v, entries in order, the loads of four entries in flight together; an
// FMA step issues only if some lane needs it.  A lane whose row has ended stays at its
// end (k1) while others go on, and indices are unsigned: none passes 2^31 + 3, and a
// matrix of up to 2^31 - 1 entries is read in bounds.
__device__ __forceinline__ double csr_dot(const int32_t *__restrict__ ci, const double *__restrict__ av,
                                          const double *__restrict__ v, unsigned k0, unsigned k1) {
    double s = 0.0;
    const unsigned lanes = __activemask();
#pragma unroll 1
    while (__any_sync(lanes, k0 < k1)) {
        int c[4];
        double a[4], g[4];
#pragma unroll
        for (int q = 0; q < 4; q++)
            if (k0 + q < k1) { c[q] = ld_stream(ci + k0 + q); a[q] = ld_stream(av + k0 + q); }
#pragma unroll
        for (int q = 0; q < 4; q++) if (k0 + q < k1) g[q] = __ldg(v + c[q]);
#pragma unroll
        for (int q = 0; q < 4; q++) {
            if (!__any_sync(lanes, k0 + q < k1)) break;
            if (k0 + q < k1) s = fma(a[q], g[q], s);
        }
        k0 = min(k0 + 4, k1);
    }
    return s;
}

// Tests on bit patterns: an FP64 comparison or conversion costs the FP64 pipe as
// much as an FMA, and the kernel is bound by that pipe.
__device__ __forceinline__ unsigned long long mag_bits(double v) { return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffULL; }
__device__ __forceinline__ bool is_nan(double v) { return mag_bits(v) > 0x7ff0000000000000ULL; }
// |v| cut to FP32 (relative error < 2^-23), or NaN outside [2^-100, 2^100)
__device__ __forceinline__ float mag_float(double v) {
    const unsigned hi = (unsigned)__double2hiint(v) & 0x7fffffffu, lo = (unsigned)__double2loint(v);
    if (hi - ((1023u - 100u) << 20) >= (200u << 20)) return __int_as_float(0x7fc00000);
    return __uint_as_float(((hi - ((1023u - 127u) << 20)) << 3) | (lo >> 29));
}

// The largest |r| / d, exactly, with few FP64 divisions (each a long FP64
// sequence).  A thread keeps its row of the largest FP32 estimate; rows whose
// estimate is within its error of that, or has none (zero rows aside), divide at
// once; at the end the rows within the error of the CTA's largest estimate do.
struct MaxQuotient {
    double mx = 0.0, r = 0.0, d = 1.0;
    float e = 0.0f;
    __device__ __forceinline__ void add(double r2, double d2) {
        if (mag_bits(r2) == 0 && !is_nan(d2) && mag_bits(d2) != 0) return;
        float e2;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(e2) : "f"(mag_float(d2)));
        e2 *= mag_float(r2);
        if (!(e2 < e * 0.99999f)) {
            if (e2 > e * 1.00001f && e2 >= 0.0f && !is_neg(d2)) { r = r2; d = d2; e = e2; }
            else {   // a NaN that the device made has its sign set, which nnmax would take for less than zero
                const double t = fabs(r2) / d2;
                mx = nnmax(mx, is_nan(t) ? __longlong_as_double(0x7ff8000000000000LL) : t);
            }
        }
    }
    __device__ __forceinline__ double finish(int *best) {
        const int top = __reduce_max_sync(0xffffffffu, __float_as_int(e));
        if ((threadIdx.x & 31) == 0) atomicMax(best, top);
        __syncthreads();
        if (e > 0.0f && e >= __int_as_float(*(volatile int *)best) * 0.99999f) mx = nnmax(mx, fabs(r) / d);
        return mx;
    }
};

// Sums of three slots and the maximum of a fourth (non-negative values) over the
// CTA, in a fixed order, to out[0 .. 4).  The sums share their shuffles: after
// two exchanges a lane holds one slot's partial sum of four lanes.
__device__ __forceinline__ void kkt_block_sum(double a0, double a1, double a2, double mx, double *out) {
    __shared__ double sh[kThreads / 32][4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // lanes with bit 4 set keep slots 1 and (none), the others 0 and 2
    const bool up = lane & 16;
    double k0 = up ? a1 : a0;
    const double s0 = up ? a0 : a1;
    k0 += __shfl_xor_sync(0xffffffffu, s0, 16);
    double k2 = a2 + __shfl_xor_sync(0xffffffffu, a2, 16);
    // lanes with bit 3 set keep slot 2, the others slot 0 or 1
    const bool up2 = lane & 8;
    double v = (up2 ? k2 : k0) + __shfl_xor_sync(0xffffffffu, up2 ? k0 : k2, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = nnmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) { sh[warp][0] = v; sh[warp][3] = mx; }
    if (lane == 16) sh[warp][1] = v;
    if (lane == 8) sh[warp][2] = v;
    __syncthreads();
    if (threadIdx.x < 4) {
        double t = sh[0][threadIdx.x];
        for (int w = 1; w < kThreads / 32; w++) t = threadIdx.x == 3 ? nnmax(t, sh[w][threadIdx.x]) : t + sh[w][threadIdx.x];
        out[threadIdx.x] = t;
    }
    __syncthreads();
}

// records [0, n) of kNoAllocSlots values summed by warp 0 in a fixed order; every
// lane gets the sums (lane l adds records l / 8, l / 8 + 4, ... of slot l % 8)
__device__ __forceinline__ double kkt_sum_records(const double *rec, int n, int stride) {
    const int slot = threadIdx.x % kNoAllocSlots;
    const bool mx = slot == RPU || slot == RDU;
    double v = 0.0;
    for (int k0 = threadIdx.x / kNoAllocSlots; k0 < n; k0 += 16) {
        double t[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            t[q] = 0.0;
            if (k0 + 4 * q < n) t[q] = __ldcg(rec + (size_t)(k0 + 4 * q) * stride + slot);
        }
#pragma unroll
        for (int q = 0; q < 4; q++) v = mx ? nnmax(v, t[q]) : v + t[q];
    }
#pragma unroll
    for (int o = kNoAllocSlots; o < 32; o <<= 1) {
        const double w = __shfl_xor_sync(0xffffffffu, v, o);
        v = mx ? nnmax(v, w) : v + w;
    }
    return v;
}

// CTA b < nbr: rows [per b, ...); else columns.  The last CTA of each group to end
// adds the group's records, the last group's adds those and writes the result.
// Bound by the FP64 pipe and by latency (6,049-bus LP: the pipe is busy 70 % of
// 96 us before the last two changes): so one launch instead of two, four entries'
// loads of a row in flight together, FP64 instructions only for the products and
// sums (bit tests for every comparison, a vote skips a warp's terms that are exact
// zeros) and about one division per CTA instead of one per row and column.
// 6,049 buses: 150.9 -> 87.4 us, 30 buses: 26.6 -> 12.4 us per call; 84.6 with non-finite
// reduced costs in a branch of their own (as selects in one line 91.5).
__global__ void __launch_bounds__(kThreads, kNoAllocCtas) k_kkt_noalloc(uc_device_lp lp, int nbr, int per, const double *__restrict__ x,
                                                          const double *__restrict__ y, double omega, int ticket,
                                                          double *__restrict__ out) {
    __shared__ double rec[kNoAllocSlots], sum[4];
    __shared__ int best;
    __shared__ bool last;
    if (threadIdx.x == 0) best = 0;
    if (threadIdx.x < kNoAllocSlots) rec[threadIdx.x] = 0.0;
    __syncthreads();
    double a0 = 0.0, a1 = 0.0, a2 = 0.0;
    MaxQuotient quot;
    const bool rows = (int)blockIdx.x < nbr;
    if (rows) {                    // |r|^2, q.y, largest unscaled residual
        const int b0 = blockIdx.x * per, b1 = min(lp.m, b0 + per);
        for (int i = b0 + threadIdx.x; i < b1; i += kThreads) {
            const int k0 = __ldg(lp.A_rowptr + i), k1 = __ldg(lp.A_rowptr + i + 1);
            const double qi = ld_stream(lp.q + i), d = ld_stream(lp.Dr + i), yi = __ldg(y + i);
            double r = csr_dot(lp.A_colidx, lp.A_val, x, k0, k1) - qi;
            if (i >= lp.m_eq && !is_neg(r) && !is_nan(r)) r = 0.0;   // min(r, 0) that keeps a NaN
            a0 = fma(r, r, a0);
            if (__any_sync(__activemask(), mag_bits(qi) != 0 || !is_fin(yi))) a1 = fma(qi, yi, a1);
            quot.add(r, d);
        }
    } else {                       // |rd|^2, c.x, bound part, largest unscaled reduced-cost residual
        const int b0 = ((int)blockIdx.x - nbr) * per, b1 = min(lp.n, b0 + per);
        for (int j = b0 + threadIdx.x; j < b1; j += kThreads) {
            const int k0 = __ldg(lp.AT_rowptr + j), k1 = __ldg(lp.AT_rowptr + j + 1);
            const double cj = ld_stream(lp.c + j), lj = ld_stream(lp.l + j), uj = ld_stream(lp.u + j);
            const double d = ld_stream(lp.Dc + j), xj = __ldg(x + j);
            const double lm = cj - csr_dot(lp.AT_colidx, lp.AT_val, y, k0, k1);
            const bool lf = is_fin(lj), uf = is_fin(uj);
            // reduced cost inside the cone the bounds allow (lp_j) and the rest, rd = lm - lp_j,
            // by sign tests; of an lm that is not finite by the subtraction (inf - inf is NaN)
            double rd, lp_j = 0.0;
            if (lf && uf) {
                if (!is_nan(lm)) lp_j = lm;
                rd = is_fin(lm) ? 0.0 : __longlong_as_double(0x7ff8000000000000LL);
            } else if (!is_fin(lm)) {
                if (!is_nan(lm)) lp_j = lf ? pos_part(lm) : uf ? neg_part(lm) : 0.0;
                rd = lm - lp_j;
            } else {
                lp_j = lf ? pos_part(lm) : uf ? neg_part(lm) : 0.0;
                rd = lf ? neg_part(lm) : uf ? pos_part(lm) : lm;
            }
            const double bound = is_neg(lp_j) ? (uf ? uj : 0.0) : (lf ? lj : 0.0);
            const unsigned lanes = __activemask();
            if (__any_sync(lanes, mag_bits(rd) != 0)) a0 = fma(rd, rd, a0);
            if (__any_sync(lanes, mag_bits(cj) != 0 || !is_fin(xj))) a1 = fma(cj, xj, a1);
            if (__any_sync(lanes, mag_bits(lp_j) != 0 && (mag_bits(bound) != 0 || !is_fin(lp_j)))) a2 = fma(bound, lp_j, a2);
            quot.add(rd, d);
        }
    }
    kkt_block_sum(a0, a1, a2, quot.finish(&best), sum);
    if (threadIdx.x == 0) {
        rec[rows ? RP2 : RD2] = sum[0];
        rec[rows ? QY : CX] = sum[1];
        if (!rows) rec[BND] = sum[2];
        rec[rows ? RPU : RDU] = sum[3];
    }
    __syncthreads();
    const int group = (int)blockIdx.x / kNoAllocGroup, ngroups = ((int)gridDim.x + kNoAllocGroup - 1) / kNoAllocGroup;
    double *mine = g_kkt_scratch + (size_t)group * kNoAllocGroup * kNoAllocSlots;   // the group's records, its sum over the first
    if (threadIdx.x < kNoAllocSlots)
        __stcg(mine + (size_t)(blockIdx.x % kNoAllocGroup) * kNoAllocSlots + threadIdx.x, rec[threadIdx.x]);
    if (threadIdx.x >= 32) return;
    const int in_group = min(kNoAllocGroup, (int)gridDim.x - group * kNoAllocGroup);
    auto ended = [&](unsigned *count, int of) {   // warp 0: whether this arrival is the last of `of`
        __threadfence();
        __syncwarp();
        if (threadIdx.x == 0) last = atomicInc(count, (unsigned)(of - 1)) == (unsigned)(of - 1);
        __syncwarp();
        __threadfence();
        return (bool)*(volatile bool *)&last;
    };
    if (!ended(&g_kkt_ended[ticket][1 + group], in_group)) return;
    const double t = kkt_sum_records(mine, in_group, kNoAllocSlots);
    __syncwarp();
    if (threadIdx.x < kNoAllocSlots) __stcg(mine + threadIdx.x, t);
    if (!ended(&g_kkt_ended[ticket][0], ngroups)) return;
    const double v = kkt_sum_records(g_kkt_scratch, ngroups, kNoAllocGroup * kNoAllocSlots);
    double T[kNoAllocSlots];
#pragma unroll
    for (int s = 0; s < kNoAllocSlots; s++) T[s] = __shfl_sync(0xffffffffu, v, s);
    if (threadIdx.x != 0) return;
    const double pobj = T[CX], dobj = T[QY] + T[BND], gap = pobj - dobj;
    out[0] = T[RPU] / (1.0 + lp.q_inf);
    out[1] = T[RDU] / (1.0 + lp.c_inf);
    out[2] = fabs(gap) / (1.0 + fabs(pobj) + fabs(dobj));
    out[3] = kkt_w(T[RP2], T[RD2], gap, omega);
    out[4] = pobj;
    out[5] = dobj;
    out[6] = T[RPU];
    out[7] = 0.0;
}

// ---------------------------------------------------------------------------
// ||A||_2 for presolve on the device: power iteration on A^T A
// ---------------------------------------------------------------------------
// A step is two launches: t = scale A w, then w = A^T t with |w| and the stopping
// test by the CTA that ends last.  The iterate is kept in the range by a power of two
// instead of divided by its norm: exact, so v = scale w loses nothing, and lambda =
// |A^T A v| / |v| with |v| = scale |w|.  Every kernel returns at once when done is set,
// so a fixed number of launches can be queued and the host only polls.
//
// Four entries' loads at a time; the first four and the row pointers come before the
// wait for the kernel before (programmatic dependent launch).  3,000 buses of 48
// periods (948 k rows and columns, 1.3 M entries): 33 us per step; as two products
// of one entry at a time, a norm by one CTA and a pass of divisions 46.  Small LPs 9 us
// (launches), large ones are bound by the gathers, which the presolved order spreads
// over L2: neither more threads per SM (64 warps 33.6) nor smaller CTAs (33.0) matter.
struct PwState {
    double lambda, prev, scale, vnorm;   // last estimates; of the current iterate
    int done;                            // 0 running, 1 converged, 2 lambda == 0
    unsigned ended;                      // CTAs of the norm that ended (wraps to zero)
};
constexpr int kPwThreads = 256;

// sum over the CTA, valid in thread 0: warp shuffles, then the warps in order
__device__ __forceinline__ double pw_block_sum(double v, double *sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = sh[0];
    if (threadIdx.x == 0)
        for (int w = 1; w < kPwThreads / 32; w++) t += sh[w];
    return t;
}

// one thread per row; NORM: y = M x and the step's norm, else y = scale M x
template <bool NORM>
__global__ void __launch_bounds__(kPwThreads) k_pw_spmv(const int32_t *__restrict__ rp, const int32_t *__restrict__ ci,
                                                        const double *__restrict__ val, int rows, const double *x, double *y,
                                                        double *part, PwState *st, double tol) {
    const int i = blockIdx.x * kPwThreads + threadIdx.x;
    // Entries left, counted down below zero while the warp's longest row lasts (to -2^31 at
    // most); k0 is used only while some are left.  32 registers and 31.9-32.2 us per step at
    // 3,000 buses; with the row's end kept and k0 held there 39 and 32.5.
    unsigned k0 = 0;
    int left = 0, c[4];
    double a[4], s = 0.0;
    if (i < rows) { k0 = rp[i]; left = rp[i + 1] - rp[i]; }
#pragma unroll
    for (int q = 0; q < 4; q++) if (q < left) { c[q] = ld_stream(ci + k0 + q); a[q] = ld_stream(val + k0 + q); }
    pdl_wait();
    pdl_trigger();
    if (__ldcg(&st->done)) return;
#pragma unroll 1
    while (__any_sync(0xffffffffu, left > 0)) {
        double g[4];
#pragma unroll
        for (int q = 0; q < 4; q++) if (q < left) g[q] = x[c[q]];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            if (!__any_sync(0xffffffffu, q < left)) break;
            if (q < left) s = fma(a[q], g[q], s);
        }
        k0 += 4;
        left -= 4;
#pragma unroll
        for (int q = 0; q < 4; q++) if (q < left) { c[q] = ld_stream(ci + k0 + q); a[q] = ld_stream(val + k0 + q); }
    }
    if (!NORM) {
        if (i < rows) y[i] = s * __ldcg(&st->scale);
        return;
    }
    if (i < rows) y[i] = s;
    __shared__ double sh[kPwThreads / 32];
    __shared__ bool last;
    const double mine = pw_block_sum(s * s, sh);
    if (threadIdx.x == 0) {
        __stcg(part + blockIdx.x, mine);
        __threadfence();
        last = atomicInc(&st->ended, gridDim.x - 1) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double t[4] = {};
    for (int p = threadIdx.x; p < (int)gridDim.x; p += 4 * kPwThreads)
#pragma unroll
        for (int q = 0; q < 4; q++)
            if (p + q * kPwThreads < (int)gridDim.x) t[q] += __ldcg(part + p + q * kPwThreads);
    const double sum = pw_block_sum((t[0] + t[1]) + (t[2] + t[3]), sh);
    if (threadIdx.x != 0) return;
    const double nrm = sqrt(sum), lam = nrm / st->vnorm;
    st->lambda = lam;
    if (lam == 0.0) st->done = 2;
    else if (fabs(lam - st->prev) <= tol * lam) st->done = 1;
    else st->prev = lam;
    const int e = max(-1000, min(1000, ((__double2hiint(nrm) >> 20) & 0x7ff) - 1023));
    st->scale = __hiloint2double((1023 - e) << 20, 0);
    st->vnorm = nrm * st->scale;
}

}  // namespace dev

int device_power_norm(const Csr &A, const Csr &AT, int max_iter, double tol, double *out) {
    using namespace dev;
    *out = 0.0;
    const int n = A.cols, m = A.rows;
    if (n == 0 || m == 0) return UC_OK;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) {
        cudaGetLastError();
        set_error("power iteration on the device: no CUDA device");
        return UC_ECUDA;
    }
    const int64_t nnz = A.nnz();
    const int np = (n + kPwThreads - 1) / kPwThreads;
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t o = off; off = align_up(off + bytes, 256); return o; };
    const size_t o_arp = take(sizeof(int32_t) * (m + 1)), o_aci = take(sizeof(int32_t) * nnz),
                 o_av = take(sizeof(double) * nnz), o_trp = take(sizeof(int32_t) * (n + 1)),
                 o_tci = take(sizeof(int32_t) * nnz), o_tv = take(sizeof(double) * nnz),
                 o_t = take(sizeof(double) * m), o_w = take(sizeof(double) * n), o_part = take(sizeof(double) * np),
                 o_st = take(sizeof(PwState));
    cudaStream_t s = nullptr;
    UC_CUDA(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
    char *D = nullptr;
    int *h_done = nullptr;
    int rc = UC_OK;
    auto fail = [&](cudaError_t e, const char *what) {
        set_error("power iteration on the device: %s failed: %s", what, cudaGetErrorString(e));
        rc = (e == cudaErrorMemoryAllocation) ? UC_ENOMEM : UC_ECUDA;
    };
    cudaError_t e = cudaMallocAsync((void **)&D, off, s);
    if (e != cudaSuccess) fail(e, "cudaMallocAsync");
    if (rc == UC_OK && (e = cudaMallocHost((void **)&h_done, sizeof(int))) != cudaSuccess) fail(e, "cudaMallocHost");
    if (rc == UC_OK) {
        std::vector<double> v0((size_t)n, 1.0 / std::sqrt((double)n));
        const PwState st0{0.0, 0.0, 1.0, 1.0, 0, 0};
        struct Up { size_t o; const void *src; size_t bytes; } ups[] = {
            {o_arp, A.rowptr.data(), sizeof(int32_t) * (m + 1)}, {o_aci, A.colidx.data(), sizeof(int32_t) * nnz},
            {o_av, A.val.data(), sizeof(double) * nnz}, {o_trp, AT.rowptr.data(), sizeof(int32_t) * (n + 1)},
            {o_tci, AT.colidx.data(), sizeof(int32_t) * nnz}, {o_tv, AT.val.data(), sizeof(double) * nnz},
            {o_w, v0.data(), sizeof(double) * n}, {o_st, &st0, sizeof(st0)}};
        for (const Up &u : ups)
            if (rc == UC_OK && (e = cudaMemcpyAsync(D + u.o, u.src, u.bytes, cudaMemcpyHostToDevice, s)) != cudaSuccess)
                fail(e, "cudaMemcpyAsync");
        // the sources are stack / local vectors: finish the copies before they go
        if (rc == UC_OK && (e = cudaStreamSynchronize(s)) != cudaSuccess) fail(e, "upload");
    }
    if (rc == UC_OK) {
        const int32_t *arp = (const int32_t *)(D + o_arp), *aci = (const int32_t *)(D + o_aci);
        const int32_t *trp = (const int32_t *)(D + o_trp), *tci = (const int32_t *)(D + o_tci);
        const double *av = (const double *)(D + o_av), *tv = (const double *)(D + o_tv);
        double *t = (double *)(D + o_t), *w = (double *)(D + o_w), *part = (double *)(D + o_part);
        PwState *st = (PwState *)(D + o_st);
        const int gm = (m + kPwThreads - 1) / kPwThreads, gn = np;
        constexpr int kPoll = 64;   // steps queued between polls of the stop flag
        for (int it = 0; it < max_iter && rc == UC_OK;) {
            const int batch = std::min(kPoll, max_iter - it);
            for (int b = 0; b < batch && e == cudaSuccess; b++) {
                e = launch_k(k_pw_spmv<false>, gm, kPwThreads, s, true, arp, aci, av, m, (const double *)w, t, (double *)nullptr, st, tol);
                if (e == cudaSuccess)
                    e = launch_k(k_pw_spmv<true>, gn, kPwThreads, s, true, trp, tci, tv, n, (const double *)t, w, part, st, tol);
            }
            if (e != cudaSuccess) { fail(e, "kernel launch"); break; }
            it += batch;
            if ((e = cudaGetLastError()) != cudaSuccess) { fail(e, "kernel launch"); break; }
            if ((e = cudaMemcpyAsync(h_done, &st->done, sizeof(int), cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
                (e = cudaStreamSynchronize(s)) != cudaSuccess) {
                fail(e, "power iteration");
                break;
            }
            if (*h_done) break;
        }
        // every pass of the loop ends with a synchronisation, so *h_done is current
        double lam = 0.0;
        if (rc == UC_OK && ((e = cudaMemcpyAsync(&lam, &st->lambda, sizeof(double), cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
                            (e = cudaStreamSynchronize(s)) != cudaSuccess))
            fail(e, "result download");
        if (rc == UC_OK) *out = (*h_done == 2) ? 0.0 : std::sqrt(lam);
    }
    if (D) cudaFreeAsync(D, s);
    cudaStreamSynchronize(s);
    if (h_done) cudaFreeHost(h_done);
    cudaStreamDestroy(s);
    return rc;
}

namespace dev {

}  // namespace dev
}  // namespace uc

using namespace uc;

extern "C" {

int uc_presolved_device_order(const uc_presolved *ps, int reorder, int32_t *prow, int32_t *pcol) {
    if (!ps || !ps->d || !prow || !pcol) { set_error("uc_presolved_device_order: null argument"); return UC_EINVAL; }
    try {
        std::vector<int32_t> r, c;
        dev::device_view(ps->d, reorder != 0, r, c);
        std::memcpy(prow, r.data(), r.size() * sizeof(int32_t));
        std::memcpy(pcol, c.data(), c.size() * sizeof(int32_t));
    } catch (const std::bad_alloc &) {
        set_error("uc_presolved_device_order: out of host memory");
        return UC_ENOMEM;
    }
    return UC_OK;
}

int uc_presolved_strided_groups(const uc_presolved *ps, int transpose, int64_t *counts, int32_t *k,
                                int32_t *off, int32_t *col, double *val) {
    if (!ps || !ps->d || !counts) { set_error("uc_presolved_strided_groups: null argument"); return UC_EINVAL; }
    try {
        std::vector<int32_t> r, c;
        const auto view = dev::device_view(ps->d, true, r, c);
        const Csr &M = transpose ? view->AT : view->A;
        const dev::StridedGroups g = dev::strided_groups(M);
        int64_t sg = 0, se = 0;
        for (size_t i = 0; i < g.k.size(); i++)
            if (g.k[i] >= 0) { sg++; se += (int64_t)g.k[i] * dev::kStrideRows; }
        counts[0] = (int64_t)g.k.size();
        counts[1] = sg;
        counts[2] = M.nnz();
        counts[3] = se;
        counts[4] = (int64_t)g.col.size();
        if (k && off && col && val) {
            std::memcpy(k, g.k.data(), g.k.size() * sizeof(int32_t));
            std::memcpy(off, g.off.data(), g.off.size() * sizeof(int32_t));
            std::memcpy(col, g.col.data(), g.col.size() * sizeof(int32_t));
            std::memcpy(val, g.val.data(), g.val.size() * sizeof(double));
        }
    } catch (const std::bad_alloc &) {
        set_error("uc_presolved_strided_groups: out of host memory");
        return UC_ENOMEM;
    }
    return UC_OK;
}

int uc_session_create(const uc_presolved *const *ps, int k, const uc_solve_opts *opts, void *stream,
                      uc_session **out) {
    if (!ps || !out || k < 1) { set_error("uc_session_create: bad arguments"); return UC_EINVAL; }
    uc_solve_opts o;
    uc_default_solve_opts(&o);
    if (opts) o = *opts;
    std::vector<const PsData *> v(k);
    std::vector<std::shared_ptr<const PsData>> own(k);
    for (int i = 0; i < k; i++) {
        if (!ps[i]) { set_error("uc_session_create: null LP %d", i); return UC_EINVAL; }
        v[i] = ps[i]->d.get();
        own[i] = ps[i]->d;
    }
    return dev::session_create(v.data(), own.data(), k, o, (cudaStream_t)stream, out);
}

int uc_session_reset(uc_session *s, int i) {
    if (!s) { set_error("uc_session_reset: null session"); return UC_EINVAL; }
    return dev::session_reset(*s, i);
}

int uc_session_run(uc_session *s, int max_replays, int *n_running) {
    if (!s) { set_error("uc_session_run: null session"); return UC_EINVAL; }
    int rc = dev::session_run(*s, max_replays > 0 ? max_replays : dev::max_replays(*s));
    if (n_running) {
        int r = 0;
        for (int i = 0; i < s->k; i++)
            if (s->active[i] && (s->h_status[i] == dev::RUNNING || s->h_status[i] == dev::NEEDS_INIT)) r++;
        *n_running = r;
    }
    if (rc) return rc;
    return s->host_status;
}

int uc_session_status(const uc_session *s, int i) {
    if (!s || i < 0 || i >= s->k) { set_error("uc_session_status: bad arguments"); return UC_EINVAL; }
    if (!s->active[i]) return 1;                           // idle
    switch (s->h_status[i]) {
        case dev::RUNNING: case dev::NEEDS_INIT: return 2;  // still iterating
        case dev::OPTIMAL: return UC_OK;
        case dev::ITER_LIMIT: return UC_EITERLIMIT;
        case dev::NUMERIC: return UC_ENUMERIC;
        case dev::INFEASIBLE: return UC_EINFEASIBLE;
        case dev::STALLED: return UC_ECUDA;
        default: return 1;
    }
}

int uc_session_result(uc_session *s, int i, uc_result **out) {
    if (!s || !out) { set_error("uc_session_result: null argument"); return UC_EINVAL; }
    return dev::session_result(*s, i, out);
}

int uc_session_set_start(uc_session *s, int i, const double *x, const double *y, double omega) {
    if (!s) { set_error("uc_session_set_start: null session"); return UC_EINVAL; }
    return dev::session_set_start(*s, i, x, y, omega);
}

int uc_session_update_lp(uc_session *s, int i, const uc_presolved *ps) {
    if (!s || !ps) { set_error("uc_session_update_lp: null argument"); return UC_EINVAL; }
    try {
        return dev::session_update_lp(*s, i, ps->d);
    } catch (const std::bad_alloc &) {
        set_error("out of host memory");
        return UC_ENOMEM;
    }
}

int uc_session_wait_limit(uc_session *s, unsigned polls) {
    if (!s || !s->block || s->k != 1 || s->vb != 64 || s->blk_threads > dev::kSmallThreads) {
        set_error("uc_session_wait_limit: needs a resident session of one small LP with FP64 values");
        return UC_EINVAL;
    }
    UC_CUDA(cudaStreamSynchronize(s->s));
    s->plan.polls = polls;
    UC_CUDA(cudaFuncSetAttribute(dev::block_kernel(*s, s->blk_threads), cudaFuncAttributeMaxDynamicSharedMemorySize, s->blk_smem_max));
    const std::vector<char> tabled = s->tabled;
    return dev::retable(*s, tabled);   // the graphs hold the plan
}

size_t uc_session_device_bytes(const uc_session *s) { return s ? s->bytes : 0; }

int uc_kkt_noalloc(const uc_device_lp *lp, const double *x, const double *y, double omega, double *out,
                   void *stream) {
    if (!lp || !x || !y || !out) { set_error("uc_kkt_noalloc: null argument"); return UC_EINVAL; }
    if (lp->n < 0 || lp->m < 0 || lp->m_eq < 0 || lp->m_eq > lp->m || !(omega > 0.0)) {
        set_error("uc_kkt_noalloc: need n, m >= 0, 0 <= m_eq <= m and omega > 0");
        return UC_EINVAL;
    }
    // block counts in 64 bits: n and m near INT_MAX must be refused, not wrap
    const int64_t nbr64 = ((int64_t)lp->m + dev::kNoAllocRows - 1) / dev::kNoAllocRows;
    const int64_t nbc64 = ((int64_t)lp->n + dev::kNoAllocRows - 1) / dev::kNoAllocRows;
    if (nbr64 + nbc64 > dev::kNoAllocMaxBlocks) {
        set_error("uc_kkt_noalloc: LP too large for the fixed scratch: ceil(m/1024) + ceil(n/1024) = %lld > %d "
                  "(n + m up to about 8.4 million)", (long long)(nbr64 + nbc64), dev::kNoAllocMaxBlocks);
        return UC_EINVAL;
    }
    int sms = 0, dev_id = 0;
    UC_CUDA(cudaGetDevice(&dev_id));
    UC_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev_id));
    int per = dev::kNoAllocSmall;
    int64_t nbr, nbc;
    for (;; per *= 2) {
        nbr = ((int64_t)lp->m + per - 1) / per;
        nbc = ((int64_t)lp->n + per - 1) / per;
        if (per == dev::kNoAllocRows || nbr + nbc <= (int64_t)dev::kNoAllocCtas * sms) break;
    }
    static std::atomic<unsigned> calls{0};
    const int ticket = (int)(calls.fetch_add(1, std::memory_order_relaxed) % dev::kNoAllocTickets);
    // an LP without rows and columns still writes its result
    const int blocks = (int)std::max<int64_t>(1, nbr + nbc);
    dev::k_kkt_noalloc<<<blocks, dev::kThreads, 0, (cudaStream_t)stream>>>(*lp, (int)nbr, per, x, y, omega, ticket, out);
    UC_CUDA(cudaGetLastError());
    return UC_OK;
}

void uc_session_free(uc_session *s) { delete s; }

int uc_solve(const uc_presolved *ps, const uc_solve_opts *opts, void *stream, uc_result **out) {
    if (!ps || !out) { set_error("uc_solve: null argument"); return UC_EINVAL; }
    *out = nullptr;
    return uc_solve_batch(&ps, 1, opts, stream, out);
}

namespace uc {
namespace dev {

// Primal feasibility polishing of the LPs of a finished session whose result
// met the relative KKT tolerance but violates a row by more than tol_abs_feas
// (absolute, unscaled): on the device their objective is cleared (c = 0), they
// restart from the result's primal point with a zero dual and the final
// primal weight, and iterate until the largest absolute row violation of the
// map output is at most tol_abs_feas (or polish_max_iter iterations).  The
// polished primal replaces the result's; its dual is kept, and the result's
// KKT figures are evaluated again for the combined point.  The session's c is
// left cleared: it is used for nothing afterwards.
static int session_polish(uc_session &X, std::vector<uc_result *> &res) {
    std::vector<int> todo;
    for (int i = 0; i < X.k; i++)
        if (res[i] && res[i]->stats.status == UC_OK && res[i]->stats.abs_primal > X.o.tol_abs_feas) todo.push_back(i);
    for (int i = 0; i < X.k; i++)
        if (res[i]) { res[i]->stats.abs_primal_unpolished = res[i]->stats.abs_primal; res[i]->stats.polish_iters = 0; }
    if (todo.empty()) return UC_OK;
    const int main_iter = X.o.max_iter;
    X.o.max_iter = X.o.polish_max_iter ? X.o.polish_max_iter : 10000;
    X.polish_tol = X.o.tol_abs_feas;
    int rc = UC_OK;
    for (int i : todo) {
        const size_t cx = X.coff[i] * 8, nx = (X.coff[i + 1] - X.coff[i]) * 8;
        if (nx && cudaMemsetAsync(X.D + X.L.c + cx, 0, nx, X.s) != cudaSuccess) { rc = UC_ECUDA; break; }
        rc = session_set_start(X, i, res[i]->x_ret.data(), nullptr, res[i]->stats.omega);
        if (rc) break;
        rc = session_reset(X, i);
        if (rc) break;
    }
    if (!rc) rc = session_run(X, max_replays(X));
    for (int i : todo) {
        if (rc) break;
        uc_result *pr = nullptr;
        const int st = session_result(X, i, &pr);
        if (!pr) { rc = st; break; }
        std::unique_ptr<uc_result> g(pr);
        uc_result &r = *res[i];
        r.stats.polish_iters = pr->stats.iters;
        if (st == UC_OK) {   // the polish reached the tolerance
            r.x_ret = pr->x_ret;
            const PsData &p = *X.P[i];
            double pobj, dobj;
            uc::host_kkt(p, r.x_ret.data(), r.y_ret.data(), r.stats.rel_primal, r.stats.rel_dual, r.stats.rel_gap,
                     r.stats.abs_primal, pobj, dobj);
            r.stats.dual_objective = dobj + p.obj_const;
        }
        r.stats.kernel_launches = pr->stats.kernel_launches;
        r.stats.solve_ms += pr->stats.solve_ms;
        r.stats.d2h_bytes += pr->stats.d2h_bytes;
    }
    X.o.max_iter = main_iter;
    X.polish_tol = 0.0;
    return rc;
}

}  // namespace dev
}  // namespace uc

int uc_solve_batch(const uc_presolved *const *ps, int k, const uc_solve_opts *opts, void *stream,
                   uc_result **outs) {
    if (!ps || !outs || k < 1) { set_error("uc_solve_batch: bad arguments"); return UC_EINVAL; }
    for (int i = 0; i < k; i++) outs[i] = nullptr;
    uc_session *s = nullptr;
    int rc = uc_session_create(ps, k, opts, stream, &s);
    if (rc) return rc;
    std::unique_ptr<uc_session> guard(s);
    rc = uc_session_reset(s, -1);
    if (rc) return rc;
    rc = dev::session_run(*s, dev::max_replays(*s));
    if (rc) return rc;
    int overall = UC_OK;
    for (int i = 0; i < k; i++) {
        int st = dev::session_result(*s, i, &outs[i]);
        if (!outs[i]) return st;
        if (st != UC_OK && overall == UC_OK) overall = st;
    }
    if (s->o.polish) {
        std::vector<uc_result *> res(outs, outs + k);
        rc = dev::session_polish(*s, res);
        if (rc) return rc;
    }
    return overall;
}

}  // extern "C"
