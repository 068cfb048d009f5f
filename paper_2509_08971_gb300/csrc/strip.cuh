// Stage update of 1D and 2D meshes: one warp per strip of cells, no shared
// memory and no block barrier.
//
// Lane l of a warp holds cell xs - 2 + l of a row: a strip is STRIP = 28 cells
// with two halo cells on each side (the boundary map applied lane by lane).
// A row's x part stays inside the warp: the slope of each cell, the face on
// its left and the flux difference take their neighbours' values by shuffles.
// Along y the warp walks its rows with the stencil in registers (last row,
// last difference, pending lower state, last face flux), so a cell is
// converted, limited and differenced once per axis and every face evaluated
// once, by one warp; two rows of warm-up and two of look-ahead per chunk.
// A row's last cells take a strip of their own; where they are twelve or fewer, a
// warp on a long walk takes several of its row chunks side by side (strip_plan), so a row
// of 29 cells costs 28 + 5 lanes, not 64: a step of 50000 rows of 29 cells 121 -> 81 us
// (block tiles: 96), FP64 5.97 -> 3.25 ms (5.05); 2048 batched problems of 29 to 32
// cells a side, five steps, 0.80 -> 0.62 ms (0.62).
//
// What bounds it: instruction issue in FP32, the FP64 pipe in FP64, and on
// small meshes the latency of one strip.  It replaces a 32 x 8 tile per block
// (primitives and both face fluxes through shared memory, two barriers, every
// slope twice): 757 issue slots per cell-stage there.  Measured, bit-identical: 4096 batched
// problems, five steps, 15.45 -> 10.07 ms; 100 FP64 steps of a 400-cell mesh
// (15 SMs instead of 4) 4.73 -> 3.09 ms; 50 FP32 steps at 256^2 0.92 -> 0.84 ms.
//
// strip_rows evaluates the same expressions in the same order whatever the
// rows per warp, so a problem of a batch equals the same mesh advanced alone
// bit for bit.
#pragma once
#include "pdl.h"
#include "stage_kernel.cuh"

namespace hh {

constexpr int STRIP = 28;                  // cells of a warp's strip (32 lanes, 4 of halo)
constexpr unsigned FULL = 0xffffffffu;

// D = -(F_{i+1/2} - F_{i-1/2}) / dx of the row whose primitives the lanes
// hold (valid in lanes 2 .. 29).
template <typename T, int PX>
__device__ __forceinline__ void strip_x(const StageArgs<T>& A, const T W[NF], T D[NF]) {
    T qL[NF], qR[NF], Fl[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        const T dm = W[f] - __shfl_up_sync(FULL, W[f], 1);
        const T s = minmod(dm, __shfl_down_sync(FULL, dm, 1));
        qR[f] = sub_half(W[f], s);
        qL[f] = __shfl_up_sync(FULL, add_half(W[f], s), 1);
    }
    hllc_axis<PX>(qL, qR, A.gamma, A.gm1, A.igm1, Fl);
#pragma unroll
    for (int f = 0; f < NF; ++f)
        D[f] = sub_over_dx(T(0), __shfl_down_sync(FULL, Fl[f], 1) - Fl[f], A.dxk[0]);
}

// Rows [y0, y1) of the strip at xs, of which the warp walks `rows` (as many, or more
// where lanes have chunks of their own, past whose end the boundary map returns cells
// nobody uses); pos: the lane's place in the strip.  RR > 0: RR rows, every load
// issued before any arithmetic and the rows unrolled (small meshes: one memory
// round trip); RR = 0: a walk of any length with the next row's loads in
// flight.  1D: y0 = 0, y1 = 1, RR = 1.
template <typename T, int DIM, int PX, int PY, int RR>
__device__ __forceinline__ void strip_rows(const StageArgs<T>& A, int xs, int pos, int y0, int y1,
                                           int rows, TileAcc<T>& acc) {
    const int n0 = A.n[0], gx = xs - 2 + pos;
    bool flx;
    const int sx = bc_map(gx, n0, A.bc_lo[0], A.bc_hi[0], flx);
    const bool own = pos >= 2 && pos < 2 + STRIP && gx < n0;
    const long long N = A.N;
    const T* const Uc = A.Uc + sx;
    const T* const U0 = A.U0 + (own ? gx : 0);
    const T dt = (T)(A.dt_dev ? *A.dt_dev : A.dt);
    const bool two = A.stage == 2;

    // conserved state of row j through the boundary map; fly: normal momentum
    // along y changes sign
    auto fetch = [&](int j, T U[NF], bool& fly) {
        fly = false;
        const int sy = DIM >= 2 ? bc_map(j, A.n[1], A.bc_lo[1], A.bc_hi[1], fly) : 0;
        const T* p = Uc + (long long)sy * n0;
#pragma unroll
        for (int f = 0; f < NF; ++f) U[f] = p[f * N];
    };
    auto prim = [&](T U[NF], bool fly, T W[NF]) {
        if (flx) U[1 + PX] = -U[1 + PX];
        if (DIM >= 2 && fly) U[1 + PY] = -U[1 + PY];
        cons_to_prim(U, A.gm1, W);
        acc.bad |= nonphys(W);
    };
    // row k of the strip completes with flux difference L
    auto finish = [&](int k, const T L[NF], const T uc[NF], const T u0[NF]) {
        T Uo[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f)
            Uo[f] = two ? add_half(T(0.5) * madd(dt, L[f], uc[f]), u0[f]) : madd(dt, L[f], uc[f]);
        if (!own || k >= y1) return;
        T* o = A.Uo + (long long)k * n0 + gx;
#pragma unroll
        for (int f = 0; f < NF; ++f) o[f * N] = Uo[f];
        if (A.rate_slot) {
            T W[NF];
            cons_to_prim(Uo, A.gm1, W);
            const T r = cell_rate(W, A.gamma, A.act, A.rdx);
            acc.rate_max = (r > acc.rate_max || r != r) ? r : acc.rate_max;
        }
        if (A.tot_partial) {
#pragma unroll
            for (int f = 0; f < NF; ++f) acc.tot[f].add(Uo[f]);
        }
    };
    auto fetch0 = [&](int k, T u0[NF]) {
        if (!two) return;
        const T* p = U0 + (long long)min(k, A.n[1] - 1) * n0;
#pragma unroll
        for (int f = 0; f < NF; ++f) u0[f] = p[f * N];
    };

    if constexpr (DIM == 1) {
        T U[NF], W[NF], D[NF], u0[NF] = {};
        bool fly;
        fetch(0, U, fly);
        fetch0(0, u0);
        prim(U, fly, W);
        strip_x<T, PX>(A, W, D);
        finish(0, D, U, u0);
    } else {
        // the column's stencil: primitives q of the last row, its difference
        // d to the row below, the lower state qL of the face above the row
        // before it, the flux F of the face below that row and its x
        // difference D; conserved values of the last two rows
        T q[NF], d[NF], qL[NF], F[NF], D[NF], Ua[NF], Ub[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) q[f] = d[f] = qL[f] = F[f] = D[f] = Ua[f] = Ub[f] = T(0);
        // Row r (cnt = r - (y0 - 2)) arrives: x part of row r-1, the face
        // between r-2 and r-1, and row r-2 completes.
        auto row = [&](int r, int cnt, T U[NF], bool fly, const T u0[NF]) {
            T W[NF], dc[NF], qR[NF], qLn[NF], Fn[NF], Dn[NF];
            T Uraw[NF];
#pragma unroll
            for (int f = 0; f < NF; ++f) Uraw[f] = U[f];
            prim(U, fly, W);
            if (cnt >= 3 && cnt < rows + 3) strip_x<T, PX>(A, q, Dn);
            if (cnt >= 1) {
#pragma unroll
                for (int f = 0; f < NF; ++f) dc[f] = W[f] - q[f];
            }
            if (cnt >= 2) {
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    const T s = minmod(d[f], dc[f]);
                    qR[f] = sub_half(q[f], s);
                    qLn[f] = add_half(q[f], s);
                }
                if (cnt >= 3) {
                    hllc_axis<PY>(qL, qR, A.gamma, A.gm1, A.igm1, Fn);
                    if (cnt >= 4) {
                        T L[NF];
#pragma unroll
                        for (int f = 0; f < NF; ++f) L[f] = sub_over_dx(D[f], Fn[f] - F[f], A.dxk[1]);
                        finish(r - 2, L, Ua, u0);
                    }
#pragma unroll
                    for (int f = 0; f < NF; ++f) {
                        F[f] = Fn[f];
                        D[f] = Dn[f];
                    }
                }
#pragma unroll
                for (int f = 0; f < NF; ++f) qL[f] = qLn[f];
            }
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                if (cnt >= 1) d[f] = dc[f];
                q[f] = W[f];
                Ua[f] = Ub[f];
                Ub[f] = Uraw[f];
            }
        };
        if constexpr (RR > 0) {
            T U[RR + 4][NF], u0[RR][NF] = {};
            bool fl[RR + 4];
#pragma unroll
            for (int i = 0; i < RR + 4; ++i) fetch(y0 - 2 + i, U[i], fl[i]);
#pragma unroll
            for (int i = 0; i < RR; ++i) fetch0(y0 + i, u0[i]);
#pragma unroll
            for (int i = 0; i < RR + 4; ++i) row(y0 - 2 + i, i, U[i], fl[i], u0[i >= 4 ? i - 4 : 0]);
        } else {
            T Un[NF];
            bool fn;
            fetch(y0 - 2, Un, fn);
#pragma unroll 1       // by two: 4096 batched problems 10.53 ms, one by one 10.40
            for (int cnt = 0; cnt < rows + 4; ++cnt) {
                const int r = y0 - 2 + cnt;
                T U[NF], u0[NF] = {};
                const bool fl = fn;
#pragma unroll
                for (int f = 0; f < NF; ++f) U[f] = Un[f];
                if (cnt < rows + 3) fetch(r + 1, Un, fn);
                if (cnt >= 4) fetch0(r - 2, u0);
                row(r, cnt, U, fl, u0);
            }
        }
    }
}

// Warp `item` of the plan p: a full strip of one of `chunks` chunks of `len` rows
// (x fastest), or `groups` chunks of the last cells' strip.  I: a type that holds
// the number of items.
template <typename T, int PX, int PY, int RR, typename I>
__device__ __forceinline__ void strip_item(const StageArgs<T>& A, const StripPlan& p, I item,
                                           int chunks, int len, TileAcc<T>& acc) {
    const int n1 = A.n[1];
    const I full = (I)p.full * chunks;
    int pos = threadIdx.x & 31, c, xs, rows;
    if (item < full) {
        c = (int)(item / (I)p.full);
        xs = (int)(item - (I)c * p.full) * STRIP;
        rows = min(len, n1 - c * len);
    } else {
        const int g = pos / p.width, first = (int)(item - full) * p.groups;
        c = min(first + g, chunks - 1);
        xs = p.full * STRIP;
        rows = min(len, n1 - first * len);             // of the first chunk, the longest
        pos = g < p.groups && first + g < chunks ? pos - g * p.width : 0;   // place 0 is a halo cell's
    }
    const int y0 = c * len;
    strip_rows<T, 2, PX, PY, RR>(A, xs, pos, y0, min(y0 + len, n1), rows, acc);
}

// Block reductions of what the block's warps accumulated: the non-physical
// flag, the rate maximum, and the block's row of the totals partial array.  Blocks
// of many warps send one atomic to the rate slot, which takes about one a
// nanosecond from the whole chip; the small blocks of small meshes need not wait.
template <typename T, int NWARP, bool ERR>
__device__ __forceinline__ void strip_epilogue(const StageArgs<T>& A, const TileAcc<T>& acc) {
    constexpr bool COMBINE = NWARP > 2;
    __shared__ double red_tot[NWARP][NF];
    __shared__ unsigned long long red_rate[NWARP];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool any_bad = __any_sync(FULL, acc.bad);
    if (any_bad && lane == 0) atomicOr(A.status, 1);
    if (A.rate_slot) {
        unsigned long long b = rate_bits(acc.rate_max);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long v = __shfl_xor_sync(FULL, b, o);
            b = v > b ? v : b;
        }
        if (lane == 0) {
            if (COMBINE) red_rate[warp] = b;
            else atomicMax(A.rate_slot, b);
        }
    }
    if (A.tot_partial) {
        const double s = warp_totals<ERR>(acc.tot, lane);
        if (sum5_writer(lane)) red_tot[warp][sum5_field(lane)] = s;
    }
    if (A.tot_partial || (COMBINE && A.rate_slot)) {
        if (NWARP > 1) __syncthreads();
        else __syncwarp();
    }
    if (COMBINE && A.rate_slot && threadIdx.x == 0) {
        unsigned long long b = red_rate[0];
        for (int w = 1; w < NWARP; ++w) b = red_rate[w] > b ? red_rate[w] : b;
        atomicMax(A.rate_slot, b);
    }
    if (A.tot_partial && threadIdx.x < NF) {
        double t = 0.0;
        for (int w = 0; w < NWARP; ++w) t += red_tot[w][threadIdx.x];
        A.tot_partial[(long long)blockIdx.x * NF + threadIdx.x] = t;
    }
}

// One strip of A.zchunk rows per warp, x fastest.
template <typename T, int DIM, int PX, int PY, int RR, int NWARP>
__global__ void __launch_bounds__(32 * NWARP) strip_kernel(const StageArgs<T> A) {
    griddep_wait();
    const long long item = (long long)blockIdx.x * NWARP + (threadIdx.x >> 5);
    TileAcc<T> acc;
    if constexpr (DIM == 1) {
        if (item * STRIP < A.n[0])
            strip_rows<T, DIM, PX, PY, RR>(A, (int)item * STRIP, threadIdx.x & 31, 0, 1, 1, acc);
    } else {
        const StripPlan p = strip_plan(A.n[0], RR == 0);
        const int chunks = (A.n[1] + A.zchunk - 1) / A.zchunk;
        if (item < strip_warps<long long>(p, chunks)) strip_item<T, PX, PY, RR>(A, p, item, chunks, A.zchunk, acc);
    }
    strip_epilogue<T, NWARP, (DIM > 1)>(A, acc);
}

}  // namespace hh
