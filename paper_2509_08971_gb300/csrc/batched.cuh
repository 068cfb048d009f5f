// Batched persistent stage kernel: many independent 1D and 2D problems of
// uneven size in one launch.
//
// Every block is persistent: it takes the next problem from a queue (one
// atomic counter over a largest-first order, so no block ever waits) and runs
// all of that problem's steps by itself:
//     r = block max of the signal rate of U          (first step only)
//     repeat nsteps times:
//         dt = cfl / r                                 (FP64)
//         stage 1 over the problem's tiles: U -> W
//         stage 2 over the problem's tiles: (U, W) -> U, signal rate fused
//         r = block max of that rate;  t += dt         (FP64)
// A problem's cells are evaluated by strip_rows, as on a single 1D or 2D mesh,
// so a problem advanced here matches the same problem advanced alone bit for
// bit: the block's warps take strips of 28 cells by a chunk of rows.  A block
// never waits on another block: problems are disjoint and the rate reduction is
// block-local.
//
// What bounds it: instruction issue (strip.cuh).  The FP64 scalars of a
// problem (widths, dt, t) are one thread's work: a warp's FP64 instruction
// holds the SM's pipe for 16 clocks.
#pragma once
#include "launch.h"
#include "strip.cuh"

namespace hh {

template <typename T>
struct BatchArgs {
    T* U;                              // packed states, updated in place
    T* W;                              // packed intermediate stage (same layout)
    const BatchProblem* probs;
    const int* order;                  // queue order (largest problems first)
    int nprob;
    int nsteps;
    double cfl;
    double* t;                         // per-problem time, FP64, advanced in place
    int* counter;                      // queue head, zeroed before the launch
    int* status;
};

// What a problem's stages share, set up once by one thread.
template <typename T>
struct BatchScalars {
    T gamma, gm1, igm1;
    width_t<T> dx, dy;
};

template <typename T>
__device__ __forceinline__ StageArgs<T> batch_stage_args(const BatchProblem& P,
                                                        const BatchScalars<T>& S, T* U, T* W,
                                                        int stage, double dt) {
    StageArgs<T> A;
    A.U0 = U;
    A.Uc = stage == 1 ? U : W;
    A.Uo = stage == 1 ? W : U;
    A.N = (long long)P.nx * P.ny;
    A.n[0] = P.nx;
    A.n[1] = P.ny;
    A.n[2] = 1;
    for (int a = 0; a < 3; ++a) {
        A.bc_lo[a] = P.bc;
        A.bc_hi[a] = P.bc;
    }
    A.gamma = S.gamma;
    A.gm1 = S.gm1;
    A.igm1 = S.igm1;
    A.dxk[0] = A.rdx[0] = S.dx;
    A.dxk[1] = A.rdx[1] = S.dy;
    A.dxk[2] = A.rdx[2] = S.dy;                       // inactive
    A.act[0] = true;
    A.act[1] = P.ny > 1;
    A.act[2] = false;
    A.dt = dt;
    A.dt_dev = nullptr;
    A.stage = stage;
    A.zchunk = 1;
    A.zlo = 0;
    A.zhi = 1;
    A.rate_slot = nullptr;
    A.tot_partial = nullptr;
    A.status = nullptr;
    A.tmap = nullptr;
    return A;
}

// The warps' largest rates into red[] (NaN propagates); the caller's barrier
// orders them before the thread that combines them.
template <typename T>
__device__ __forceinline__ void warp_rate_max(T r, unsigned long long* red) {
    unsigned long long b = rate_bits(r);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long v = __shfl_xor_sync(FULL, b, o);
        b = v > b ? v : b;
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = b;
}

// NW warps per block; 16 warps per SM (128 registers a thread).  FP32: of 24, 80
// registers, the walk spills, 10.5 -> 17.9 ms.  FP64 spills ~560 bytes here; with the 252
// registers that it wants, 8 warps per SM, 256 2D problems of 32 to 128 cells a side
// take 9.5 ms against 16.3, but 8192 1D ones of 16 to 64 cells 2.55 against 1.43.
template <typename T, int NW>
__global__ void __launch_bounds__(32 * NW, 16 / NW) batched_kernel(const BatchArgs<T> B) {
    constexpr int NT = 32 * NW;
    __shared__ unsigned long long red[NW];
    __shared__ BatchScalars<T> s_sc;
    __shared__ double s_dt, s_t;
    __shared__ int s_next, s_chunks, s_len;
    const int tid = threadIdx.x, warp = tid >> 5;
    bool bad = false;

    // dt of the next step from the rates in red[], by one thread; every step
    // but the last advances t
    auto next_dt = [&]() {
        unsigned long long m = 0;
        for (int w = 0; w < NW; ++w) m = red[w] > m ? red[w] : m;
        const double rate = __longlong_as_double((long long)m);
        const bool ok = rate > 0.0 && !isinf(rate);
        s_dt = ok ? B.cfl / rate : 0.0;
        return ok;
    };

    for (;;) {
        __syncthreads();
        if (tid == 0) s_next = atomicAdd(B.counter, 1);
        __syncthreads();
        const int qi = s_next;
        if (qi >= B.nprob) break;
        const BatchProblem P = B.probs[B.order[qi]];
        T* U = B.U + P.off;
        T* W = B.W + P.off;
        const bool two_d = P.ny > 1;
        const long long N = (long long)P.nx * P.ny;
        const int strips = (P.nx + STRIP - 1) / STRIP;   // 1D
        const StripPlan plan = two_d ? strip_plan(P.nx, true) : StripPlan{strips, 0, 0};
        if (tid == 0) {
            s_sc.gamma = (T)P.gamma;
            s_sc.gm1 = (T)(P.gamma - 1.0);
            s_sc.igm1 = (T)(1.0 / (P.gamma - 1.0));
            s_sc.dx = make_width<T>(1.0 / P.nx);
            s_sc.dy = make_width<T>(1.0 / P.ny);
            s_t = B.t[B.order[qi]];
        }
        if (two_d && warp == NW - 1) {
            // row chunks per strip: of 1 .. 32, the one whose rounds over the
            // block's warps take the fewest rows (a chunk pays about three
            // rows for its warm-up and look-ahead)
            const int k = (tid & 31) + 1;
            const long long cost = (long long)((strip_warps<unsigned>(plan, k) + NW - 1) / NW) * ((P.ny + k - 1) / k + 3);
            const unsigned key = ((unsigned)min(cost, (1ll << 25) - 1) << 6) | (unsigned)k;
            const unsigned best = __reduce_min_sync(FULL, key);
            if ((tid & 31) == 0) {
                const int c = (int)(best & 63u);
                s_len = (P.ny + c - 1) / c;
                s_chunks = (P.ny + s_len - 1) / s_len;           // without empty ones
            }
        }
        __syncthreads();
        const BatchScalars<T> sc = s_sc;
        const int chunk = s_len, chunks = s_chunks;              // 2D: rows of a chunk, chunks
        const unsigned items = two_d ? strip_warps<unsigned>(plan, chunks) : 0;   // at most 32 chunks: below 2^32

        // signal rate of the initial state
        {
            const StageArgs<T> A = batch_stage_args<T>(P, sc, U, W, 1, 0.0);
            T r0 = T(0);
            for (long long c = tid; c < N; c += NT) {
                T Uc[NF], Wp[NF];
#pragma unroll
                for (int f = 0; f < NF; ++f) Uc[f] = U[f * N + c];
                cons_to_prim(Uc, A.gm1, Wp);
                bad |= nonphys(Wp);
                const T r = cell_rate(Wp, A.gamma, A.act, A.rdx);
                r0 = (r > r0 || r != r) ? r : r0;
            }
            warp_rate_max(r0, red);
        }
        __syncthreads();
        for (int step = 0; step < B.nsteps; ++step) {
            if (tid == 0) {
                if (!next_dt()) bad = true;
                s_t += s_dt;
            }
            __syncthreads();
            const double dt = s_dt;
            TileAcc<T> acc;
#pragma unroll 1
            for (int stage = 1; stage <= 2; ++stage) {
                StageArgs<T> A = batch_stage_args<T>(P, sc, U, W, stage, dt);
                // non-null: strip_rows folds the signal rate of the new state
                // into acc (it never writes through the pointer)
                A.rate_slot = stage == 2 ? red : nullptr;
                if (two_d) {
                    for (unsigned it = warp; it < items; it += NW)
                        strip_item<T, 0, 1, 0>(A, plan, it, chunks, chunk, acc);
                } else {
                    for (int it = warp; it < strips; it += NW)
                        strip_rows<T, 1, 0, 0, 1>(A, it * STRIP, tid & 31, 0, 1, 1, acc);
                }
                if (stage == 2) warp_rate_max(acc.rate_max, red);
                __syncthreads();            // every cell of this stage written
            }
            bad |= acc.bad;
        }
        if (tid == 0) B.t[B.order[qi]] = s_t;
    }
    if (__syncthreads_or(bad) && tid == 0) atomicOr(B.status, 1);
}

}  // namespace hh
