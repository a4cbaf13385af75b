// step_weak.cu -- the symmetric FP64 step whose weakly perturbed pairs take
// the short solve of kepler_weak.cuh (the FP64 form, the double-word form and
// the mixed form under the literal rule; order 2), on the systolic tiles of
// step_sym.cu and in the row-group layout of step_grp.cu.
//
// A warp solves a tile in systolic steps: lane l owns row l and at step k
// holds the pair with column (l + k) mod 32, the column's sums travelling
// from lane to lane by shuffles.  The lanes whose pair is weak add its
// increments at once (weak_add).  The others (the strong pairs) go to the
// warp's queue in shared memory and are solved 32 at a time by the seeded
// FP64 solver, so that a rare close pair does not make its warp run a
// 75-instruction FP64 solve for one lane; a step with more than
// kWeakInline strong lanes solves them at once.  Steps whose pairs are strong
// in larger part than that pays for take the kernels that solve every pair
// (step_sym.cu, step_grp.cu, step_df64.cu): both are launched, and the prep
// kernel's choice (sample_classes) lets one of them return at once, 1 us per
// step.  Separations out of the class's range, us per step with this kernel
// alone -> so: 8192 bodies FP64 8000 -> 5220, double-word 6680 -> 2230; 2999
// bodies 1105 -> 766, double-word 949 -> 351.
//
// Bound: the FP64 pipe (16 FP64 instructions per pair and 16 cycles each)
// and the issue slots (966 instructions per pair and warp) nearly alike: ncu
// at 8192 bodies (black hole), 70 % and 62 %, neither full with the 12 warps
// per SM that 168 registers leave.  ms per step: 16384 bodies (black hole)
// 20.36 -> 5.16 in row groups; Plummer 1024 0.109 -> 0.043, 2048 0.358 ->
// 0.103, 4000 1.30 -> 0.313 (the kernels of step_sym.cu and step_grp.cu with
// the seed before); the double-word form, 16384 bodies with binaries: 8.29 ->
// 5.46 (step_df64.cu before: every pair in 1922 double-word flops); the mixed
// form's literal rule, 5003 bodies: 2.11 -> 0.57; the default guess, 2999
// bodies, a fourth-order step on host arrays: 3.26 -> 0.75; the learned
// guess, 8192 bodies with binaries: 7.06 -> 1.62.
#include <cuda_runtime.h>

#include "kepler_df64.cuh"
#include "kepler_fp64.cuh"
#include "kepler_weak.cuh"
#include "pair_batch_fp64.cuh"
#include "step_common.cuh"
#include "step_grp.cuh"
#include "step_weak.cuh"
#include "weak_rows.cuh"

namespace sakura {

// Strong lanes of a step that are queued at most.  Solved in place, more lanes
// than these take a batch for themselves, at most 32 / 9 times what they take
// in the queue; steps with as many are rare in the runs that take this kernel
// (prep_weak_kernel chooses the others where one pair in six is strong).
constexpr int kWeakInline = 8;
// entries of a warp's queue on tiles: a segment's, and a rest below one batch
constexpr int kWeakQueue = 32 * kWeakInline + 31;

__device__ __forceinline__ dw split_dw(double x)
{
    const float h = __double2float_rn(x);
    return {h, __double2float_rn(x - (double)h)};
}

// The forms: FP64 with the single-precision seed; double-word; mixed under
// the literal rule (e_max < 1), seeded; FP64 with an analytic guess; FP64
// with the network's guess.
constexpr int kWeakFp64 = 0, kWeakDf64 = 1, kWeakMixed = 2, kWeakGuess = 3, kWeakLearned = 4;

// Solve counts of a lane: evaluations, bisections, Taylor carries, pairs
// (double-word form) or ordered pairs (mixed form) solved on the FP32 pipe.
struct StrongCount {
    int iters, fb, carried, n32;
};

// Solve of 32 strong pairs (i, j), one per lane, from the drifted state; the
// increments over m to out[lane][0..5], m_j and -m_i to [6] and [7] (their
// products are formed by the FMAs that add them to the sums).  FP64: the FP64
// solver, seeded from the float copy of the state.  Double-word: the
// double-word solver for the pairs it admits, the FP64 solver from the
// analytic guess for the others; its operands are converted on the integer
// pipe (with conversion instructions, as many as 42 FP64-pipe instructions of
// a pair, and products of their own a step of 800 bodies whose pairs are all
// strong took 110 us, now 81; FP64 124 -> 112).  Mixed: the FP32 solver for
// the pairs its class rule admits, the seeded FP64 solver for the others.
// Guess, learned: the FP64 iteration from that guess (the network's weights
// read from global memory: a batch in a hundred steps or so needs them).
template <int MODE>
__device__ __noinline__ StrongCount weak_strong_solve(const StepArgs &a, bool valid, int i, int j,
                                                      int weight, double (*out)[12],
                                                      unsigned *status)
{
    constexpr bool DW = MODE == kWeakDf64;
    constexpr bool SEED = MODE == kWeakFp64 || MODE == kWeakMixed;
    const int lane = threadIdx.x & 31;
    const int64_t n = a.n;
    const double *X = a.X;
    const KeplerParams kp{a.tol, a.max_iter, a.bisection};
    StrongCount cnt{0, 0, 0, 0};
    double rr[3], vv[3], mi = 0.0, mj = 0.0;
    if (valid) {
        mi = X[6 * n + i];
        mj = X[6 * n + j];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            rr[q] = X[q * n + i] - X[q * n + j];
            vv[q] = X[(3 + q) * n + i] - X[(3 + q) * n + j];
        }
    }
    bool need64 = valid;
    double d[6];
    if (DW) {
        dw r[3], v[3], m = {0.0f, 0.0f}, dd[6];
        K32 o;
        o.ok = false;
        o.x = o.s = 0.0f;
        o.iters = 0;
        if (valid) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                r[q] = dw_from_double(rr[q]);
                v[q] = dw_from_double(vv[q]);
            }
            m = dw_from_double(mi + mj);
            o = dw_phase1(r, v, m, a.ptau32, a.t32, a.guess);
        }
        const bool big = __any_sync(0xffffffffu, o.ok && fabsf(o.x) > 0x1p-8f);
        int evals = 0;
        const bool solved = o.ok && dw_phase2(r, v, m, split_dw(a.pre * a.tau), split_dw(a.tau),
                                              split_dw(a.post * a.tau), o.s, big, dd, evals);
        if (solved) {
#pragma unroll
            for (int q = 0; q < 6; ++q) d[q] = dw_double(dd[q]);
        }
        need64 = valid && !solved;
        cnt.iters = o.iters + evals;
        cnt.n32 = solved;
    }
    if (MODE == kWeakMixed && valid) {
        const float *X32 = a.X32;
        float hi[2][3], lo[2][3], v[2][3], d32[6];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            hi[0][q] = X32[q * n + i];
            lo[0][q] = X32[(3 + q) * n + i];
            v[0][q] = X32[(6 + q) * n + i];
            hi[1][q] = X32[q * n + j];
            lo[1][q] = X32[(3 + q) * n + j];
            v[1][q] = X32[(6 + q) * n + j];
        }
        Pair32 pr;
        pair32_setup(pr, hi[0], lo[0], v[0], X32[9 * n + i], hi[1], lo[1], v[1], X32[9 * n + j],
                     a.rule);
        int it32 = 0;
        if (pr.fp32 && pair32_solve(pr, a.t32, a.post32, a.guess, d32, it32)) {
#pragma unroll
            for (int q = 0; q < 6; ++q) d[q] = (double)d32[q];
            need64 = false;
            cnt.n32 = weight;
        }
    }
    if (!DW || __any_sync(0xffffffffu, need64)) {
        PairSolve p;
        if (need64) {
            pair_setup(p, a.tau, mi + mj, rr[0], rr[1], rr[2], vv[0], vv[1], vv[2], a.pre,
                       SEED ? -1 : (MODE == kWeakLearned ? 2 : a.guess));
            if (SEED) {
                const float *X32 = a.X32;
                float dr[3], dv[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    dr[q] = __fadd_rn(__fsub_rn(X32[q * n + i], X32[q * n + j]),
                                      __fsub_rn(X32[(3 + q) * n + i], X32[(3 + q) * n + j]));
                    dv[q] = __fsub_rn(X32[(6 + q) * n + i], X32[(6 + q) * n + j]);
                }
                const K32 o =
                    k32_phase1(dr, dv, X32[9 * n + i] + X32[9 * n + j], a.ptau32, a.t32, 2);
                if (o.ok && dbits(p.t) == dbits(a.tau) && !p.done) {
                    p.s = f2d(o.s);
                } else if (!p.done) {
                    p.s = p.t * p.ir0;
                    const double cq = 0.5 * p.s * (p.eta0 * p.ir0);
                    if (magbits(cq) < 0x3fe0000000000000LL) p.s = fma(-cq, p.s, p.s);
                }
            }
        } else {
            p.done = true;
            p.beta = p.s = 0.0;
            p.iters = 0;
            p.status = 0;
            p.carried = false;
        }
        // the batch's result rows serve as the network's staging before them
        if (MODE == kWeakLearned)
            learned_guess_warp(p, need64, *a.mlp, reinterpret_cast<__nv_bfloat16 *>(out));
        double d64[6];
        int iters = 0;
        fp64_solve_warp<SEED>(p, need64, a.tau, a.post * a.tau, kp, d64, iters, cnt.fb);
        cnt.iters += iters;
        if (need64) {
#pragma unroll
            for (int q = 0; q < 6; ++q) d[q] = d64[q];
            *status |= p.status;
            cnt.carried = p.carried;
        }
    }
    if (valid) {
#pragma unroll
        for (int q = 0; q < 6; ++q) out[lane][q] = d[q];
        out[lane][6] = mj;
        out[lane][7] = -mi;
    }
    return cnt;
}

// Ordered pairs that a queue entry stands for: one on a diagonal tile, whose
// two orders are separate entries, else two.
__device__ __forceinline__ int strong_weight(int2 q)
{
    return (q.x >> 5) == ((q.y & 0xffffff) >> 5) ? 1 : 2;
}

// Per-warp state of the weak pair kernels.
struct WeakWarp {
    int2 *queue;              // [kWeakQueue] strong pairs: i, j | tag << 24
    double (*sacc)[32];       // [12][32] sums of the tile's inline strong solves
    double (*res)[12];        // [32][12] results of a batch of strong solves
    int tail;
    unsigned status;
    long long it_sum, slots, fallbacks, carries, n32;
    int it_max;

    template <bool STATS>
    __device__ __forceinline__ void count(int lane, const StrongCount &c)
    {
        if (STATS) {
            it_sum += c.iters;
            fallbacks += c.fb;
            carries += c.carried;
            n32 += c.n32;
            it_max = max(it_max, c.iters);
            const int wmax = __reduce_max_sync(0xffffffffu, c.iters);
            if (lane == 0) slots += 32LL * wmax;
        }
    }

    template <bool STATS>
    __device__ __forceinline__ void finish(const StepArgs &a, int lane)
    {
        status = __reduce_or_sync(0xffffffffu, status);
        if (lane == 0 && status) atomicOr(a.status, status);
        if (STATS) {
            for (int o = 16; o > 0; o >>= 1) {
                it_sum += __shfl_xor_sync(0xffffffffu, it_sum, o);
                slots += __shfl_xor_sync(0xffffffffu, slots, o);
                fallbacks += __shfl_xor_sync(0xffffffffu, fallbacks, o);
                carries += __shfl_xor_sync(0xffffffffu, carries, o);
                n32 += __shfl_xor_sync(0xffffffffu, n32, o);
                it_max = max(it_max, __shfl_xor_sync(0xffffffffu, it_max, o));
            }
            if (lane == 0) {
                atomicAdd(&a.stats[kStatIters], (unsigned long long)it_sum);
                atomicAdd(&a.stats[kStatSlots], (unsigned long long)slots);
                atomicAdd(&a.stats[kStatFallbacks], (unsigned long long)fallbacks);
                atomicAdd(&a.stats[kStatCarries], (unsigned long long)carries);
                atomicAdd(&a.stats[kStatFp32Pairs], (unsigned long long)n32);
                atomicMax(&a.stats[kStatMaxIters], (unsigned long long)it_max);
            }
        }
    }
};

// Steps k0 .. k1 - 1 of the tile of row block 32 I.. (lane l: row i0 + l)
// and column block 32 J.. (layout indices; L maps them to particles).
// Returns the tile's sums of the lane's row in row[0..5] and of column
// (lane + k1 - 1) mod 32 in col[0..5] (positions, then velocities).
template <bool STATS, int MODE>
__device__ __forceinline__ void weak_tile(const StepArgs &a, const WeakStep &ws, int n, bool rev,
                                          int i0, int j0, int k0, int k1, int tag, int lane,
                                          WeakWarp &s, double row[6], double col[6])
{
    const float4 *rows = ws.rows;
    const bool diag = i0 == j0;
    const int i = i0 + lane;
    const bool irow = i < n;
    const int last = n - 1;
    const int il = rev ? last - min(i, last) : min(i, last);
    const WeakParticle A =
        weak_unpack(rows[il], rows[n + il], rows[2 * n + il], rows[3 * n + il]);
    const float sa = weak_speed2(A);
    double vr[3] = {0, 0, 0}, vc[3] = {0, 0, 0};
    dw er[3], rr[3], ec[3], rc[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) er[q] = rr[q] = ec[q] = rc[q] = dw{0.0f, 0.0f};
    bool dirty = false;
    for (int k = k0; k < k1; ++k) {
        const int c = (lane + k) & 31;
        const int j = j0 + c;
        const bool valid = irow && j < n && (!diag || c != lane);
        const int jl = rev ? last - min(j, last) : min(j, last);
        const WeakParticle B =
            weak_unpack(rows[jl], rows[n + jl], rows[2 * n + jl], rows[3 * n + jl]);
        WeakDiff d;
        bool weak = weak_class(A, sa, B, d) && valid;
        // the mixed form's FP32 class holds bound pairs only (e_max < 1):
        // pairs that are not clearly unbound go to the queue, where the
        // class rule itself decides
        if (MODE == kWeakMixed) weak = weak && weak_unbound(A, sa, B, d);
        if (weak) weak_add(A, B, d, vr, er, rr, vc, ec, rc);
        const bool strong = valid && !weak;
        const unsigned mask = __ballot_sync(0xffffffffu, strong);
        if (STATS) {
            const int any = __any_sync(0xffffffffu, weak);
            s.it_sum += weak ? 1 : 0;
            (MODE == kWeakDf64 ? s.n32 : s.carries) += weak ? 1 : 0;
            s.it_max = max(s.it_max, weak ? 1 : 0);
            if (lane == 0 && any) s.slots += 32;
        }
        if (mask) {
            if (__popc(mask) <= kWeakInline) {
                if (strong)
                    s.queue[s.tail + __popc(mask & ((1u << lane) - 1u))] =
                        make_int2(i, j | (tag << 24));
                s.tail += __popc(mask);
            } else {
                if (!dirty) {
#pragma unroll
                    for (int q = 0; q < 12; ++q) s.sacc[q][lane] = 0.0;
                    dirty = true;
                    __syncwarp();
                }
                s.count<STATS>(lane, weak_strong_solve<MODE>(a, strong, rev ? last - i : i,
                                                             rev ? last - j : j, diag ? 1 : 2,
                                                             s.res, &s.status));
                if (strong) {
#pragma unroll
                    for (int q = 0; q < 6; ++q) {
                        const double x = s.res[lane][q];
                        s.sacc[q][lane] = fma(s.res[lane][6], x, s.sacc[q][lane]);
                        if (!diag) s.sacc[6 + q][c] = fma(s.res[lane][7], x, s.sacc[6 + q][c]);
                    }
                }
                __syncwarp();
            }
        }
        if (!diag && k + 1 < k1) {
            const int src = (lane + 1) & 31;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                vc[q] = __shfl_sync(0xffffffffu, vc[q], src);
                ec[q].h = __shfl_sync(0xffffffffu, ec[q].h, src);
                ec[q].l = __shfl_sync(0xffffffffu, ec[q].l, src);
                rc[q].h = __shfl_sync(0xffffffffu, rc[q].h, src);
                rc[q].l = __shfl_sync(0xffffffffu, rc[q].l, src);
            }
        }
    }
    const int c = (lane + k1 - 1) & 31;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        row[q] = dw_to_double(rr[q]);
        row[3 + q] = fma(-ws.inv_t, dw_to_double(er[q]), vr[q]);
        col[q] = -dw_to_double(rc[q]);
        col[3 + q] = fma(ws.inv_t, dw_to_double(ec[q]), -vc[q]);
    }
    if (dirty) {
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            row[q] += s.sacc[q][lane];
            col[q] += s.sacc[6 + q][c];
        }
        __syncwarp();
    }
}

// Tiles (below 4096 bodies): the partition and slots of step_sym.cu.  A
// segment's sums are written first; the results of its strong pairs are
// added to the slots afterwards, by the warp that owns them: batches of 32
// as the queue fills, and what is left at the block's end with the other
// warps' rests, packed (a warp of a 1024-body step has one or two strong
// pairs in all).
template <bool STATS, int MODE>
__global__ void __launch_bounds__(128, 3)
    pair_step_weak_kernel(StepArgs a, WeakStep ws, int Smax, int64_t T)
{
    __shared__ int2 queue[4][kWeakQueue];
    __shared__ double sacc[4][12][32];
    __shared__ double res[128][12];
    __shared__ int cnt[4];
    griddep_wait();
    if (gate_closed(a.gate)) return;
    griddep_launch();
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const int64_t n = a.n;
    const int64_t W = (int64_t)gridDim.x * 4;
    const int64_t w = (int64_t)blockIdx.x * 4 + wib;
    WeakWarp s{queue[wib], sacc[wib], res + 32 * wib, 0, 0u, 0, 0, 0, 0, 0, 0};

    // adds the results of entries e0 .. e0 + m - 1 of the queue, at
    // res[r0 ..], to their slots (written before): lane c component c
    auto add_results = [&](int e0, int m, int r0) {
        for (int e = 0; e < m; ++e) {
            const int2 q = s.queue[e0 + e];
            const int i = q.x, j = q.y & 0xffffff, h = q.y >> 24;
            const int I = i >> 5, J = j >> 5;
            if (lane < (I == J ? 6 : 12)) {
                const int64_t slot = lane < 6 ? (int64_t)J * Smax + h : (int64_t)I * Smax + h;
                const int c = lane < 6 ? lane : lane - 6;
                double *dst = a.partial + (slot * 6 + c) * n + (lane < 6 ? i : j);
                *dst = fma(res[r0 + e][lane < 6 ? 6 : 7], res[r0 + e][c], *dst);
            }
        }
    };

    const int64_t p1 = (w + 1) * T / W;
    for (int64_t pos = w * T / W; pos < p1;) {
        const int64_t tile = pos >> 5;
        const int k0 = (int)(pos & 31);
        const int k1 = p1 - pos < 32 - k0 ? k0 + (int)(p1 - pos) : 32;
        const int h = (int)(w - sym_owner(32 * tile, W, T));
        pos += k1 - k0;
        int64_t I, J;
        sym_tile_of(tile, I, J);
        double row[6], col[6];
        weak_tile<STATS, MODE>(a, ws, (int)n, false, (int)(32 * I), (int)(32 * J), k0, k1, h, lane, s,
                         row, col);
        // row sums of rows i to slot (J, h); column sums to slot (I, h)
        const int64_t i = 32 * I + lane, j = 32 * J + ((lane + k1 - 1) & 31);
        if (i < n) {
            double *dst = a.partial + (J * Smax + h) * 6 * n;
#pragma unroll
            for (int q = 0; q < 6; ++q) dst[q * n + i] = row[q];
        }
        if (I != J && j < n) {
            double *dst = a.partial + (I * Smax + h) * 6 * n;
#pragma unroll
            for (int q = 0; q < 6; ++q) dst[q * n + j] = col[q];
        }
        __syncwarp();
        while (s.tail >= 32) {
            s.tail -= 32;
            const int2 q = s.queue[s.tail + lane];
            s.count<STATS>(lane, weak_strong_solve<MODE>(a, true, q.x, q.y & 0xffffff,
                                                         strong_weight(q), s.res, &s.status));
            __syncwarp();
            add_results(s.tail, 32, 32 * wib);
            __syncwarp();
        }
    }
    // the rests of the block's four queues, packed into batches
    if (lane == 0) cnt[wib] = s.tail;
    __syncthreads();
    const int c0 = cnt[0], c1 = c0 + cnt[1], c2 = c1 + cnt[2], tot = c2 + cnt[3];
    if (32 * wib < tot) {
        const int e = 32 * wib + lane;
        const bool v = e < tot;
        const int o = e < c0 ? 0 : (e < c1 ? 1 : (e < c2 ? 2 : 3));
        const int b0 = o == 0 ? 0 : (o == 1 ? c0 : (o == 2 ? c1 : c2));
        const int2 q = v ? queue[o][e - b0] : make_int2(0, 0);
        s.count<STATS>(lane,
                       weak_strong_solve<MODE>(a, v, q.x, q.y & 0xffffff, strong_weight(q), s.res,
                                               &s.status));
    }
    __syncthreads();
    add_results(0, s.tail, wib == 0 ? 0 : (wib == 1 ? c0 : (wib == 2 ? c1 : c2)));
    s.finish<STATS>(a, lane);
}

// The row-group layout (grp_layout.cuh), from 4096 bodies: a block of G = 4
// warps sweeps windows of 2 phases, warp w taking row block w of the group
// in every phase (a heavy particle's pairs are mostly weak and cost what the
// others' do, so the row blocks need not rotate over the warps as in
// step_grp.cu, and a warp keeps one row sum per component instead of G).
// The column blocks are read through L1, which the small shared memory (58
// KB per block) leaves room for: with rotating rows (78 KB) the step took
// 6.11 ms at 16384 bodies, this way 5.18; one block of 12 warps per SM 5.43,
// two of 6 5.36, four of 3 5.27.
// The strong pairs of a window are solved together by the block, packed
// into batches of 32, between the window's barriers; each warp adds its own
// pairs' results to its own sums in queue order (deterministic).
constexpr int kWeakGrpWindow = 2;
constexpr size_t weak_grp_smem()
{
    return sizeof(double) * kFp64GrpWarps * 32 *
               (6 * kWeakGrpWindow + 6 + 12 + 12) +
           sizeof(int2) * kFp64GrpWarps * (32 * kWeakInline * kWeakGrpWindow);
}

template <bool STATS, int MODE>
__global__ void __launch_bounds__(kFp64GrpWarps * 32, 3)
    pair_step_grp_weak_kernel(StepArgs a, WeakStep ws, GrpLayout L, GrpParts parts)
{
    constexpr int G = kFp64GrpWarps;
    constexpr int WIN = kWeakGrpWindow;
    // column sums of the window's tiles, row sums of the group, inline sums
    // and batch results per warp, then the warps' queues
    extern __shared__ __align__(16) unsigned char gsm[];
    double(*cs)[WIN][6][32] = reinterpret_cast<double(*)[WIN][6][32]>(gsm);
    double(*rs)[6][32] = reinterpret_cast<double(*)[6][32]>(cs + G);
    double(*sacc)[12][32] = reinterpret_cast<double(*)[12][32]>(rs + G);
    double(*res)[12] = reinterpret_cast<double(*)[12]>(sacc + G);
    int2(*queue)[32 * kWeakInline * WIN] =
        reinterpret_cast<int2(*)[32 * kWeakInline * WIN]>(res + 32 * G);
    __shared__ int cnt[G];
    griddep_wait();
    if (gate_closed(a.gate)) return;
    griddep_launch();
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const int tid = threadIdx.x;
    const int64_t n = a.n;
    const int64_t nb = L.nb;
    const int64_t B = gridDim.x;
    const int64_t b = blockIdx.x;
    WeakWarp s{queue[wib], sacc[wib], res + 32 * wib, 0, 0u, 0, 0, 0, 0, 0, 0};

    GrpPos cur = grp_block_start(L, b, B);
    __shared__ GrpPos s_end;
    if (tid == 0) s_end = grp_block_start(L, b + 1, B);
    for (int e = tid; e < G * 6 * 32; e += G * 32) (&rs[0][0][0])[e] = 0.0;
    __syncthreads();
    auto in_range = [&](const GrpPos &p) {
        const GrpPos e = s_end;
        return p.g < e.g || (p.g == e.g && (p.t < e.t || (p.t == e.t && p.k < e.k)));
    };
    auto window_len = [&](const GrpPos &p) {
        const GrpPos e = s_end;
        const int64_t m = p.g < e.g ? nb - p.g * G - p.t : e.t - p.t + (e.k > 0 ? 1 : 0);
        return (int)(m < WIN ? m : WIN);
    };
    int wl = in_range(cur) ? window_len(cur) : 0;

    while (wl > 0) {
        const int64_t g = cur.g, R = grp_rows(L, g), J0 = g * G + cur.t;
        const int kfirst = cur.k;
        const int klast = (g == s_end.g && cur.t + wl - 1 == s_end.t) ? s_end.k : 32;
        for (int cb = 0; cb < wl; ++cb) {
            const int64_t t = cur.t + cb;
            const int r = wib;
            double row[6] = {0, 0, 0, 0, 0, 0}, col[6] = {0, 0, 0, 0, 0, 0};
            int c = lane;
            if (r <= t && r < R) {
                const int64_t I = g * G + r, Jt = J0 + cb;
                const int kb = cb == 0 ? kfirst : 0;
                const int ke = cb == wl - 1 ? klast : 32;
                weak_tile<STATS, MODE>(a, ws, (int)n, L.rev != 0, (int)(32 * I), (int)(32 * Jt), kb, ke,
                                 cb, lane, s, row, col);
                c = (lane + ke - 1) & 31;
                if (I == Jt) {
#pragma unroll
                    for (int q = 0; q < 6; ++q) col[q] = 0.0;
                }
#pragma unroll
                for (int q = 0; q < 6; ++q) rs[wib][q][lane] += row[q];
            }
#pragma unroll
            for (int q = 0; q < 6; ++q) cs[wib][cb][q][c] = col[q];
        }
        // the window's strong pairs, the warps' queues packed into batches;
        // each warp adds its own pairs' results to its own sums
        if (lane == 0) cnt[wib] = s.tail;
        __syncthreads();
        int base = 0, tot = 0;
#pragma unroll
        for (int w = 0; w < G; ++w) {
            if (w < wib) base += cnt[w];
            tot += cnt[w];
        }
        for (int r0 = 0; r0 < tot; r0 += 32 * G) {
            if (r0 + 32 * wib < tot) {
                const int e = r0 + 32 * wib + lane;
                const bool v = e < tot;
                int o = 0, eo = e;
                while (o + 1 < G && eo >= cnt[o]) eo -= cnt[o++];
                const int2 q = v ? queue[o][eo] : make_int2(0, 0);
                s.count<STATS>(lane, weak_strong_solve<MODE>(
                                         a, v, (int)grp_particle(L, n, q.x),
                                         (int)grp_particle(L, n, q.y & 0xffffff),
                                         strong_weight(q), s.res, &s.status));
            }
            __syncthreads();
            const int m0 = max(base, r0), m1 = min(base + s.tail, r0 + 32 * G);
            for (int e = m0; e < m1; ++e) {
                const int2 q = s.queue[e - base];
                const int i = q.x, j = q.y & 0xffffff, cb = q.y >> 24;
                const double *r = res[e - r0];
                if (lane < 6) {
                    double &x = rs[wib][lane][i & 31];
                    x = fma(r[6], r[lane], x);
                } else if (lane < 12 && (i >> 5) != (j >> 5)) {
                    double &x = cs[wib][cb][lane - 6][j & 31];
                    x = fma(r[7], r[lane - 6], x);
                }
            }
            __syncthreads();
        }
        s.tail = 0;
        GrpPos nxt{g, cur.t + wl, 0};
        if (nxt.t == nb - g * G) {
            nxt.g = g + 1;
            nxt.t = 0;
        }
        const int wln = in_range(nxt) ? window_len(nxt) : 0;
        for (int e = tid; e < wl * 192; e += G * 32) {
            const int cb = e / 192, rem = e - cb * 192, c = rem & 31, q = rem >> 5;
            double sum = cs[0][cb][q][c];
#pragma unroll
            for (int w = 1; w < G; ++w) sum += cs[w][cb][q][c];
            if (cb == 0 && kfirst > 0) {
                parts.colx[(b * 6 + q) * 32 + c] = sum;
            } else {
                const int64_t j = 32 * (J0 + cb) + c;
                if (j < n) parts.col[(g * 6 + q) * n + j] = sum;
            }
        }
        if (nxt.g != g || wln == 0) {
            const int64_t h = b - grp_owner(grp_phase_x(L, g, 0), B, L);
            double *dst = parts.row + h * 6 * n;
            for (int e = tid; e < R * 192; e += G * 32) {
                const int r = e / 192, rem = e - r * 192, l = rem & 31, q = rem >> 5;
                const int64_t i = 32 * (g * G + r) + l;
                if (i < n) dst[q * n + i] = rs[r][q][l];
                rs[r][q][l] = 0.0;
            }
        }
        __syncthreads();
        cur = nxt;
        wl = wln;
    }
    s.finish<STATS>(a, lane);
}

// Which kernels a run's steps take: those of the weak pairs, or, where more
// than limit of kWeakSample pairs of the state before the run are strong
// (under the mixed form's rule: or not certainly unbound), those that solve
// every pair.  The pairs are drawn by a hash of their number, so the choice
// depends on the state alone.  A pair per thread in 16 blocks: the test's 40
// FP64 instructions take 10 us when one block makes them all.
constexpr int kPrepThreads = 64, kSampleBlocks = kWeakSample / kPrepThreads;

__device__ __forceinline__ WeakParticle sample_particle(const double *state, const double *mass,
                                                        int64_t n, int64_t i, double tau)
{
    WeakParticle p;
    p.x = state[i];
    p.y = state[n + i];
    p.z = state[2 * n + i];
    p.mt = tau * mass[i];
#pragma unroll
    for (int q = 0; q < 3; ++q) p.w[q] = {(float)(tau * state[(3 + q) * n + i]), 0.0f};
    p.mh = {(float)(tau * p.mt), 0.0f};
    return p;
}

__device__ __forceinline__ void sample_classes(const double *state, const double *mass, int64_t n,
                                               double tau, int block, const WeakChoice &ch)
{
    uint32_t h = (uint32_t)(kPrepThreads * block + threadIdx.x + 1) * 0x9e3779b1u;
    h = (h ^ (h >> 15)) * 0x85ebca77u;
    h ^= h >> 13;
    const uint32_t g = (h * 0xc2b2ae3du) ^ (h >> 16);
    const int64_t i = (int64_t)(((uint64_t)h * (uint64_t)n) >> 32);
    int64_t j = i + 1 + (int64_t)(((uint64_t)g * (uint64_t)(n - 1)) >> 32);
    if (j >= n) j -= n;
    const WeakParticle a = sample_particle(state, mass, n, i, tau);
    const WeakParticle b = sample_particle(state, mass, n, j, tau);
    const float sa = weak_speed2(a);
    WeakDiff d;
    const bool weak = weak_class(a, sa, b, d) && (!ch.unbound || weak_unbound(a, sa, b, d));
    const unsigned strong = __syncthreads_count(!weak);
    if (threadIdx.x != 0) return;
    // the counts' sum and, above it, their number; the last block leaves zero
    const unsigned before = atomicAdd(&ch.p->sum, strong + (1u << 16));
    if (before >> 16 != kSampleBlocks - 1) return;
    ch.p->sum = 0u;
    ch.p->every = (before & 0xffffu) + strong > (unsigned)ch.limit ? 1 : 0;
}

// Eq. 27a (order 2), the drifted state with its float copy for the FP64
// solves, and the rows of the weak pairs; one thread per particle, and the
// first kSampleBlocks blocks for the choice of the kernels
__global__ void prep_weak_kernel(const double *state, const double *mass, double *X, float *X32,
                                 float4 *rows, int64_t n, double tau, unsigned *status,
                                 WeakChoice ch)
{
    griddep_launch();
    if (blockIdx.x < kSampleBlocks) {
        sample_classes(state, mass, n, tau, blockIdx.x, ch);
        return;
    }
    const int64_t i = (int64_t)(blockIdx.x - kSampleBlocks) * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double m = mass[i], drift = 0.5 * tau;
    if (!(m > 0.0)) atomicOr(status, kStatusMass);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const double x0 = state[q * n + i], v = state[(3 + q) * n + i];
        const double x = fma(v, drift, x0);
        X[q * n + i] = x;
        X[(3 + q) * n + i] = v;
        if (X32) {
            const float hi = __double2float_rn(x);
            X32[q * n + i] = hi;
            X32[(3 + q) * n + i] = __double2float_rn(x - (double)hi);
            X32[(6 + q) * n + i] = __double2float_rn(v);
        }
        if (ch.X3) tf_row_component(ch.X3, n, i, q, x, v);
        weak_row_component(rows, n, i, q, x0, v, tau);
    }
    X[6 * n + i] = m;
    if (ch.X3) tf_row_mass(ch.X3, n, i, m);
    if (X32) X32[9 * n + i] = __double2float_rn(m);
    weak_row_mass(rows, n, i, m, tau);
}

// Small systems (up to 928 bodies on 152 SMs): a step is two kernels of a few
// microseconds each, bound by the latencies of launches, loads and solves and
// not by any rate, so the chain between them is kept short.  A block takes
// 4 K consecutive tile-steps of one tile, K = 2, 4 or 8 per warp.  It
// prepares the tile's 64 particles from the state
// itself, in shared memory (no drift kernel; the solves then read shared
// memory), and adds its warps' sums there, so that it leaves one partial sum
// per tile and block: S = 32 / (4 K) slots per tile, slot (J, h) with the row
// sums of the rows' particles, slot (I, h) with the column sums of the
// columns'.  Within the block layout indices are local: rows 0 .. 31, columns
// 32 .. 63 (a diagonal tile: 0 .. 31).  PER_SM 2: up to 255 registers, no
// spills but 44 bytes of the learned guess's; 3 where the grid needs three
// blocks per SM to be resident at once.
// Four steps of a run and a copy of the state before them in us, pair kernel
// on general tiles with drift, pair and apply kernels before -> now: 128
// bodies 70 -> 43, 512 135 -> 90, 760 155 -> 114, 928 181 -> 151; where most
// pairs are strong, 128 bodies 95 -> 67 (seeded FP64; the other forms alike).
struct WeakSmallShared {
    float4 rows[4 * 64];
    double X[7 * 64];
    float X32[10 * 64];
    double sacc[4][12][32];
    double res[128][12];
    int2 queue[4][kWeakQueue];
    int cnt[4];
    StepArgs args;
};

template <bool STATS, int MODE, int PER_SM>
__global__ void __launch_bounds__(128, PER_SM)
    pair_step_weak_small_kernel(const __grid_constant__ StepArgs a, WeakSmall ws)
{
    __shared__ WeakSmallShared sh;
    constexpr bool F32 = MODE == kWeakFp64 || MODE == kWeakMixed;
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const int tid = threadIdx.x;
    const int n = (int)a.n;
    const int per = 4 * ws.steps, S = 32 / per;
    const int tile = blockIdx.x / S, h = blockIdx.x - S * tile;
    int64_t I, J;
    sym_tile_of(tile, I, J);
    const int i0 = 32 * (int)I, j0 = 32 * (int)J;
    const bool diag = I == J;
    const int nl = diag ? min(32, n - i0) : 32 + min(32, n - j0);
    griddep_wait();
    griddep_launch();
    for (int e = tid; e < 4 * 64; e += 128) {
        const int q = e >> 6, t = e & 63;
        if (t >= nl) continue;
        const int i = t < 32 ? i0 + t : j0 + t - 32;
        if (q == 3) {
            const double m = ws.mass[i];
            if (!(m > 0.0)) atomicOr(a.status, kStatusMass);
            sh.X[6 * nl + t] = m;
            if (F32) sh.X32[9 * nl + t] = __double2float_rn(m);
            weak_row_mass(sh.rows, nl, t, m, a.tau);
            continue;
        }
        const double x0 = ws.src[q * n + i], v = ws.src[(3 + q) * n + i];
        const double x = fma(v, 0.5 * a.tau, x0);
        sh.X[q * nl + t] = x;
        sh.X[(3 + q) * nl + t] = v;
        if (F32) {
            const float hi = __double2float_rn(x);
            sh.X32[q * nl + t] = hi;
            sh.X32[(3 + q) * nl + t] = __double2float_rn(x - (double)hi);
            sh.X32[(6 + q) * nl + t] = __double2float_rn(v);
        }
        weak_row_component(sh.rows, nl, t, q, x0, v, a.tau);
    }
    if (tid == 0) {
        sh.args = a;
        sh.args.X = sh.X;
        sh.args.X32 = F32 ? sh.X32 : nullptr;
        sh.args.n = nl;
    }
    __syncthreads();

    const StepArgs &b = sh.args;
    const WeakStep wl{sh.rows, ws.inv_t};
    double(*sacc)[32] = sh.sacc[wib];
    WeakWarp s{sh.queue[wib], sacc, sh.res + 32 * wib, 0, 0u, 0, 0, 0, 0, 0, 0};
    auto add_results = [&](int e0, int m, int r0) {
        for (int e = 0; e < m; ++e) {
            const int2 q = s.queue[e0 + e];
            const int i = q.x, j = q.y & 0xffffff;
            if (lane < (diag ? 6 : 12)) {
                const double *r = sh.res[r0 + e];
                double &x = sacc[lane][(lane < 6 ? i : j) & 31];
                x = fma(r[lane < 6 ? 6 : 7], r[lane < 6 ? lane : lane - 6], x);
            }
        }
    };
    {
        const int k0 = h * per + wib * ws.steps, k1 = k0 + ws.steps;
        double row[6], col[6];
        weak_tile<STATS, MODE>(b, wl, nl, false, 0, diag ? 0 : 32, k0, k1, 0, lane, s, row, col);
        const int c = (lane + k1 - 1) & 31;
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            sacc[q][lane] = row[q];
            sacc[6 + q][c] = col[q];
        }
    }
    __syncwarp();
    while (s.tail >= 32) {
        s.tail -= 32;
        const int2 q = s.queue[s.tail + lane];
        s.count<STATS>(lane, weak_strong_solve<MODE>(b, true, q.x, q.y & 0xffffff,
                                                     strong_weight(q), s.res, &s.status));
        __syncwarp();
        add_results(s.tail, 32, 32 * wib);
        __syncwarp();
    }
    // the rests of the block's four queues, packed into batches
    if (lane == 0) sh.cnt[wib] = s.tail;
    __syncthreads();
    const int c0 = sh.cnt[0], c1 = c0 + sh.cnt[1], c2 = c1 + sh.cnt[2], tot = c2 + sh.cnt[3];
    if (tot) {
        if (32 * wib < tot) {
            const int e = 32 * wib + lane;
            const bool v = e < tot;
            const int o = e < c0 ? 0 : (e < c1 ? 1 : (e < c2 ? 2 : 3));
            const int b0 = o == 0 ? 0 : (o == 1 ? c0 : (o == 2 ? c1 : c2));
            const int2 q = v ? sh.queue[o][e - b0] : make_int2(0, 0);
            s.count<STATS>(lane,
                           weak_strong_solve<MODE>(b, v, q.x, q.y & 0xffffff, strong_weight(q),
                                                   s.res, &s.status));
        }
        __syncthreads();
        add_results(0, s.tail, wib == 0 ? 0 : (wib == 1 ? c0 : (wib == 2 ? c1 : c2)));
        __syncthreads();
    }
    for (int e = tid; e < (diag ? 6 : 12) * 32; e += 128) {
        const int q = e >> 5, l = e & 31;
        const int i = (q < 6 ? i0 : j0) + l;
        const double sum = (sh.sacc[0][q][l] + sh.sacc[1][q][l]) +
                           (sh.sacc[2][q][l] + sh.sacc[3][q][l]);
        const int64_t slot = (q < 6 ? J : I) * S + h;
        if (i < n) a.partial[(slot * 6 + (q < 6 ? q : q - 6)) * n + i] = sum;
    }
    s.finish<STATS>(a, lane);
}

// Eqs. 27b-d after pair_step_weak_small_kernel: block (P, q) takes 32
// particles and the components q, 3 + q; its warps sum the slots w, w + 8,
// ... of the slots = nb S, four loads in flight, and warp 0 adds the warps'
// sums in order.  The drift is that of the pair kernel's blocks, from the
// state again.  src may be dst.
constexpr int kSmallApplyWarps = 8;

__global__ void __launch_bounds__(32 * kSmallApplyWarps)
    apply_weak_small_kernel(const double *src, double *dst, const double *partial, int n,
                            int slots, double tau, unsigned *status)
{
    __shared__ double red[kSmallApplyWarps][2][32];
    griddep_wait();
    griddep_launch();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int q = blockIdx.y;
    const int i = 32 * blockIdx.x + lane;
    double x0 = 0.0, v = 0.0;
    if (wid == 0 && i < n) {
        x0 = src[q * n + i];
        v = src[(3 + q) * n + i];
    }
    double er = 0.0, ev = 0.0;
    if (i < n) {
        const double *p = partial + q * n + i;
#pragma unroll 4
        for (int k = wid; k < slots; k += kSmallApplyWarps) {
            er += p[(int64_t)k * 6 * n];
            ev += p[((int64_t)k * 6 + 3) * n];
        }
    }
    red[wid][0][lane] = er;
    red[wid][1][lane] = ev;
    __syncthreads();
    if (wid != 0 || i >= n) return;
    double r[4], w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        r[k] = red[2 * k][0][lane] + red[2 * k + 1][0][lane];
        w[k] = red[2 * k][1][lane] + red[2 * k + 1][1][lane];
    }
    const double v1 = v + ((w[0] + w[1]) + (w[2] + w[3]));
    const double x = fma(v, 0.5 * tau, x0) + ((r[0] + r[1]) + (r[2] + r[3]));
    const double x1 = fma(v1, 0.5 * tau, x);
    if (!isfinite(x1) || !isfinite(v1)) atomicOr(status, kStatusNonfinite);
    dst[q * n + i] = x1;
    dst[(3 + q) * n + i] = v1;
}

// The state and the masses of host memory, for the blocks of the small
// kernel that each read them again.
__global__ void copy_state_kernel(const double *src, const double *mass, double *dst, double *mdst,
                                  int n)
{
    griddep_launch();
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < 6 * n)
        dst[e] = src[e];
    else if (e < 7 * n)
        mdst[e - 6 * n] = mass[e - 6 * n];
}

namespace {

template <int MODE>
const void *weak_kernel_ptr(bool stats, bool grp)
{
    if constexpr (MODE == kWeakGuess || MODE == kWeakLearned)  // without statistics only
        return grp ? (const void *)pair_step_grp_weak_kernel<false, MODE>
                   : (const void *)pair_step_weak_kernel<false, MODE>;
    else if (grp)
        return stats ? (const void *)pair_step_grp_weak_kernel<true, MODE>
                     : (const void *)pair_step_grp_weak_kernel<false, MODE>;
    else
        return stats ? (const void *)pair_step_weak_kernel<true, MODE>
                     : (const void *)pair_step_weak_kernel<false, MODE>;
}

const void *weak_kernel(bool stats, WeakForm form, bool grp)
{
    switch (form) {
    case WeakForm::Df64: return weak_kernel_ptr<kWeakDf64>(stats, grp);
    case WeakForm::Mixed: return weak_kernel_ptr<kWeakMixed>(stats, grp);
    case WeakForm::Guess: return weak_kernel_ptr<kWeakGuess>(stats, grp);
    case WeakForm::Learned: return weak_kernel_ptr<kWeakLearned>(stats, grp);
    default: return weak_kernel_ptr<kWeakFp64>(stats, grp);
    }
}

template <int MODE, int PER_SM>
const void *weak_small_ptr(bool stats)
{
    if constexpr (MODE == kWeakGuess || MODE == kWeakLearned)
        return (const void *)pair_step_weak_small_kernel<false, MODE, PER_SM>;
    else
        return stats ? (const void *)pair_step_weak_small_kernel<true, MODE, PER_SM>
                     : (const void *)pair_step_weak_small_kernel<false, MODE, PER_SM>;
}

template <int PER_SM>
const void *weak_small_kernel(bool stats, WeakForm form)
{
    switch (form) {
    case WeakForm::Df64: return weak_small_ptr<kWeakDf64, PER_SM>(stats);
    case WeakForm::Mixed: return weak_small_ptr<kWeakMixed, PER_SM>(stats);
    case WeakForm::Guess: return weak_small_ptr<kWeakGuess, PER_SM>(stats);
    case WeakForm::Learned: return weak_small_ptr<kWeakLearned, PER_SM>(stats);
    default: return weak_small_ptr<kWeakFp64, PER_SM>(stats);
    }
}

}  // namespace

void launch_pair_step_weak_small(const StepArgs &a, const WeakSmall &ws, int blocks, bool three,
                                 bool stats, WeakForm form, cudaStream_t s)
{
    void *args[] = {(void *)&a, (void *)&ws};
    launch_pdl(three ? weak_small_kernel<3>(stats, form) : weak_small_kernel<2>(stats, form),
               dim3(blocks), dim3(128), args, 0, s);
}

void launch_apply_weak_small(const double *src, double *dst, const double *partial, int n,
                             int slots, double tau, unsigned *status, cudaStream_t s)
{
    void *args[] = {(void *)&src, (void *)&dst, (void *)&partial, (void *)&n,
                    (void *)&slots, (void *)&tau, (void *)&status};
    launch_pdl((const void *)apply_weak_small_kernel, dim3((unsigned)((n + 31) / 32), 3),
               dim3(32 * kSmallApplyWarps), args, 0, s);
}

void launch_copy_state(const double *src, const double *mass, double *dst, double *mdst, int n,
                       cudaStream_t s)
{
    copy_state_kernel<<<(7 * n + 127) / 128, 128, 0, s>>>(src, mass, dst, mdst, n);
}

int pair_step_weak_blocks_per_sm(bool stats, WeakForm form)
{
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, weak_kernel(stats, form, false), 128, 0) !=
        cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return b > 0 ? b : 1;
}

void launch_pair_step_weak(const StepArgs &a, const WeakStep &ws, int Smax, int64_t T, int blocks,
                           bool stats, WeakForm form, cudaStream_t s)
{
    int Sv = Smax;
    int64_t it = T;
    void *args[] = {(void *)&a, (void *)&ws, (void *)&Sv, (void *)&it};
    launch_pdl(weak_kernel(stats, form, false), dim3(blocks), dim3(128), args, 0, s);
}

int pair_step_grp_weak_blocks_per_sm(bool stats, WeakForm form)
{
    const void *fn = weak_kernel(stats, form, true);
    int b = 0;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)weak_grp_smem()) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, fn, kFp64GrpWarps * 32,
                                                      weak_grp_smem()) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return b > 0 ? b : 1;
}

void launch_pair_step_grp_weak(const StepArgs &a, const WeakStep &ws, const GrpLayout &L,
                               const GrpParts &parts, int blocks, bool stats, WeakForm form,
                               cudaStream_t s)
{
    const void *fn = weak_kernel(stats, form, true);
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)weak_grp_smem());
    GrpLayout Lv = L;
    GrpParts pv = parts;
    void *args[] = {(void *)&a, (void *)&ws, (void *)&Lv, (void *)&pv};
    launch_pdl(fn, dim3(blocks), dim3(kFp64GrpWarps * 32), args, weak_grp_smem(), s);
}

void launch_prep_weak(const double *state, const double *mass, double *X, float *X32,
                      float4 *rows, int64_t n, double tau, unsigned *status,
                      const WeakChoice &ch, cudaStream_t s)
{
    const int threads = kPrepThreads;
    prep_weak_kernel<<<kSampleBlocks + (unsigned)((n + threads - 1) / threads), threads, 0, s>>>(
        state, mass, X, X32, rows, n, tau, status, ch);
}

}  // namespace sakura
