// Diffusion levels stored by colour.  The red-black smoother of a mesh order
// takes every second cell of a row, so each half-sweep moves the sectors of
// both colours of x and b for half of their cells.  Here the cells of colour c = (i + j + k) & 1
// of a level sit in an array of their own, cell (i, j, k) at
//   ((c n2 + k) n1 + j) stride + p,   p = i / 2,
// rows padded to a multiple of four.  In the row (j, k) of colour c the cells are i = 2p + s,
// s = (j + k + c) & 1; the neighbours of cell p along y and z have the same p
// in the other colour's rows, those along x are p and p - 1 (s = 0) or p and p + 1
// (s = 1) of the other colour's row (j, k).  Everything a half-sweep touches is
// contiguous, and a thread takes V = 16 bytes of cells with vector loads.
//
// On a periodic x axis whose rows end inside a vector, the entry after the
// row's last cell repeats its first (x and D), so that the shifted neighbours
// of a vector need no wrap of their own.  Other padding stays zero.
//
// Only for levels whose periodic axes are even (a proper two-colouring), of
// FLD_SPLIT_CELLS cells at least.
//
// What bounds it: memory.  A half-sweep of a 256^3 FP32 level moves 168 MB (x
// of one colour, b and x of the other, D of both) in 34 us against 242 MB in 52 us
// in mesh order; the prolongation corrects one colour only (19 us against 36), the
// residual norm takes 34 us (53), the step to 1e-5 (four cycles) 2.20 ms (3.11).
#pragma once
#include "pdl.h"

namespace hh {
namespace {

// Neighbour offsets of a cell along one axis (coordinate c of n cells, the
// axis' element stride): lo / hi are added to the cell's index (across the
// wrap on a periodic axis; 0 at a wall, whose face carries no flux), face
// bit 0 / 1 set when the low / high face carries a flux.
struct AxisNb {
    int lo, hi, face;
};

__device__ __forceinline__ AxisNb axis_nb(int c, int n, bool per, int stride) {
    const bool inl = c > 0, inh = c + 1 < n;
    AxisNb b;
    b.lo = inl ? -stride : (per ? (n - 1) * stride : 0);
    b.hi = inh ? stride : (per ? -(n - 1) * stride : 0);
    b.face = (inl || per ? 1 : 0) | (inh || per ? 2 : 0);
    return b;
}

template <typename T> struct VecOf;
template <> struct VecOf<float> { using type = float4; static constexpr int V = 4; };
template <> struct VecOf<double> { using type = double2; static constexpr int V = 2; };

// A level's array addressed by cell: by colour (stride > 0) or in mesh order.
template <typename T>
struct CellArray {
    T* a;
    int n0, n1, n2, stride;
    __device__ __forceinline__ int index(int i, int j, int k) const {
        if (stride == 0) return (k * n1 + j) * n0 + i;
        return ((((i + j + k) & 1) * n2 + k) * n1 + j) * stride + (i >> 1);
    }
};

template <typename T>
struct SplitArgs {
    T* x;                    // both colours
    const T* b;
    const T* D;
    int n[3];
    int h;                   // cells of a colour in an even row, (n0 + 1) / 2
    int stride;              // entries of a row
    int groups;              // vectors of a row
    int color;               // entries of one colour
    T wk[3];                 // dt / (2 dx^2) per axis (0: inactive)
    bool per[3];
};

template <typename T>
__device__ __forceinline__ void vload(const T* p, T (&v)[VecOf<T>::V]) {
    const typename VecOf<T>::type q = *reinterpret_cast<const typename VecOf<T>::type*>(p);
    v[0] = q.x;
    v[1] = q.y;
    if constexpr (VecOf<T>::V == 4) {
        v[2] = q.z;
        v[3] = q.w;
    }
}

// The cells of a row (j, k) of colour c: cells [0, cnt).
template <typename T>
__device__ __forceinline__ int row_cells(const SplitArgs<T>& a, int s) {
    return (a.n[0] - s + 1) >> 1;
}

// What the stencil of V cells p0 .. of row (j, k), colour c, reads besides the
// z neighbours and the other colour's row: all loads of one place, so that a
// caller issues them together.
template <typename T>
struct SplitRow {
    static constexpr int V = VecOf<T>::V;
    T Dc[V], b[V], xl[V], Dl[V], xh[V], Dh[V];   // own, y neighbours
    T x[V];                                      // own, where a residual is wanted
    T xe, De;                                    // the x neighbour outside the vector
    T wy[2], wz[2];                              // face weights' factor, 0 at a wall
    int s;                                       // parity
};

template <bool OWN, typename T>
__device__ __forceinline__ void split_row_load(const SplitArgs<T>& a, int c, int j, int k, int p0,
                                               SplitRow<T>& v) {
    constexpr int V = VecOf<T>::V;
    const AxisNb ny = axis_nb(j, a.n[1], a.per[1], a.stride);
    const AxisNb nz = axis_nb(k, a.n[2], a.per[2], 0);
    v.s = (j + k + c) & 1;
    v.wy[0] = ny.face & 1 ? a.wk[1] : T(0);
    v.wy[1] = ny.face & 2 ? a.wk[1] : T(0);
    v.wz[0] = nz.face & 1 ? a.wk[2] : T(0);
    v.wz[1] = nz.face & 2 ? a.wk[2] : T(0);
    const int row = (k * a.n[1] + j) * a.stride;
    const int mine = c * a.color + row, other = (1 - c) * a.color + row;
    vload(a.D + mine + p0, v.Dc);
    vload(a.b + mine + p0, v.b);
    if constexpr (OWN) vload(a.x + mine + p0, v.x);
    vload(a.x + other + ny.lo + p0, v.xl);
    vload(a.D + other + ny.lo + p0, v.Dl);
    vload(a.x + other + ny.hi + p0, v.xh);
    vload(a.D + other + ny.hi + p0, v.Dh);
    const int e = v.s ? (p0 + V < a.h ? p0 + V : (a.per[0] ? 0 : p0))
                      : (p0 > 0 ? p0 - 1 : (a.per[0] ? a.h - 1 : 0));
    v.xe = a.x[other + e];
    v.De = a.D[other + e];
}

// diag = 1 + sum w and off = sum w x_nb of the vector's cells.  Along x the
// other colour's entry p comes first, then p + 1 or p - 1; WALLS: the x axis
// ends at walls, whose faces carry nothing.
template <bool WALLS, typename T>
__device__ __forceinline__ void split_eval(const SplitArgs<T>& a, int p0, const SplitRow<T>& v,
                                           const T (&x0)[VecOf<T>::V], const T (&D0)[VecOf<T>::V],
                                           const T (&xm)[VecOf<T>::V], const T (&Dm)[VecOf<T>::V],
                                           const T (&xp)[VecOf<T>::V], const T (&Dp)[VecOf<T>::V],
                                           T (&diag)[VecOf<T>::V], T (&off)[VecOf<T>::V]) {
    constexpr int V = VecOf<T>::V;
    const bool s = v.s;
#pragma unroll
    for (int u = 0; u < V; ++u) {
        const int i = 2 * (p0 + u) + v.s;
        const T xn = s ? (u + 1 < V ? x0[u + 1 < V ? u + 1 : 0] : v.xe) : (u ? x0[u ? u - 1 : 0] : v.xe);
        const T Dn = s ? (u + 1 < V ? D0[u + 1 < V ? u + 1 : 0] : v.De) : (u ? D0[u ? u - 1 : 0] : v.De);
        // entry p is the upper neighbour of an even cell, the lower of an odd one
        const bool in = !WALLS || s || i + 1 < a.n[0];
        const bool out = !WALLS || (s ? i + 1 < a.n[0] : i > 0);
        T dg = T(1), of = T(0);
        auto add = [&](T Db, T xb, T wk) {
            const T w = (v.Dc[u] + Db) * wk;
            dg += w;
            of += w * xb;
        };
        add(D0[u], x0[u], in ? a.wk[0] : T(0));
        add(Dn, xn, out ? a.wk[0] : T(0));
        add(v.Dl[u], v.xl[u], v.wy[0]);
        add(v.Dh[u], v.xh[u], v.wy[1]);
        add(Dm[u], xm[u], v.wz[0]);
        add(Dp[u], xp[u], v.wz[1]);
        diag[u] = dg;
        off[u] = of;
    }
}

// Thread's vector column (p0, j) of a level; false past the last.
template <typename T>
__device__ __forceinline__ bool split_column(const SplitArgs<T>& a, int& p0, int& j) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    j = t / a.groups;
    p0 = (t - j * a.groups) * VecOf<T>::V;
    return j < a.n[1];
}

// The march of a vector column over planes [k0, k1): the other colour's x
// and D of the planes k - 1, k, k + 1 stay in registers, so a plane's rows are
// loaded once for the three planes that use them.  op(k, row, diag, off).
// OWN: for a residual; its extra vector leaves no registers to load a plane
// ahead, which a half-sweep does (256^3 FP32: half-sweep 45 -> 34 us with the
// loads ahead; residual norm 36 us without, 47 us with them and x not).
template <bool WALLS, bool OWN, typename T, class Op>
__device__ __forceinline__ void split_march(const SplitArgs<T>& a, int c, int p0, int j, int k0,
                                            int k1, const Op& op) {
    constexpr int V = VecOf<T>::V;
    const int oc = (1 - c) * a.color;
    auto plane = [&](int k, T (&x)[V], T (&D)[V]) {    // k through the z boundary
        if (k < 0) k = a.per[2] ? a.n[2] - 1 : 0;
        if (k >= a.n[2]) k = a.per[2] ? 0 : a.n[2] - 1;
        const int o = oc + (k * a.n[1] + j) * a.stride + p0;
        vload(a.x + o, x);
        vload(a.D + o, D);
    };
    T xm[V], Dm[V], x0[V], D0[V], xp[V], Dp[V];
    SplitRow<T> v;
    plane(k0 - 1, xm, Dm);
    plane(k0, x0, D0);
    if constexpr (!OWN) {
        plane(k0 + 1, xp, Dp);
        split_row_load<OWN>(a, c, j, k0, p0, v);
    }
#pragma unroll 1
    for (int k = k0; k < k1; ++k) {
        T xq[V], Dq[V];
        SplitRow<T> w;
        if constexpr (OWN) {
            plane(k + 1, xp, Dp);
            split_row_load<OWN>(a, c, j, k, p0, v);
        } else if (k + 1 < k1) {
            plane(k + 2, xq, Dq);
            split_row_load<OWN>(a, c, j, k + 1, p0, w);
        }
        T diag[V], off[V];
        split_eval<WALLS>(a, p0, v, x0, D0, xm, Dm, xp, Dp, diag, off);
        op(k, v, diag, off);
#pragma unroll
        for (int u = 0; u < V; ++u) {
            xm[u] = x0[u];
            Dm[u] = D0[u];
            x0[u] = xp[u];
            D0[u] = Dp[u];
        }
        if constexpr (!OWN) {
            v = w;
#pragma unroll
            for (int u = 0; u < V; ++u) {
                xp[u] = xq[u];
                Dp[u] = Dq[u];
            }
        }
    }
}

// Values of the vector's cells of a row (those past its end are padding).
template <typename T>
__device__ __forceinline__ void split_store(const SplitArgs<T>& a, int c, int j, int k, int p0,
                                            const T (&v)[VecOf<T>::V]) {
    constexpr int V = VecOf<T>::V;
    const int cnt = row_cells(a, (j + k + c) & 1);
    T* row = a.x + c * a.color + (k * a.n[1] + j) * a.stride;
    if (p0 + V <= cnt) {
        typename VecOf<T>::type q;
        q.x = v[0];
        q.y = v[1];
        if constexpr (V == 4) {
            q.z = v[2];
            q.w = v[3];
        }
        *reinterpret_cast<typename VecOf<T>::type*>(row + p0) = q;
    } else {
#pragma unroll
        for (int u = 0; u < V; ++u)
            if (p0 + u < cnt) row[p0 + u] = v[u];
    }
    if (p0 == 0 && a.per[0] && a.h < a.stride) row[a.h] = v[0];
}

// One half-sweep, colour c.
template <typename T, bool WALLS>
__global__ void __launch_bounds__(128, 4) split_smooth_kernel(const SplitArgs<T> a, int c, int chunk) {
    griddep_wait();
    if (griddep_many_blocks()) griddep_launch_dependents();
    constexpr int V = VecOf<T>::V;
    int p0, j;
    if (split_column(a, p0, j)) {
        const int k0 = blockIdx.y * chunk, k1 = min(k0 + chunk, a.n[2]);
        split_march<WALLS, false>(a, c, p0, j, k0, k1,
                    [&](int k, const SplitRow<T>& v, const T (&diag)[V], const T (&off)[V]) {
                        T x[V];
#pragma unroll
                        for (int u = 0; u < V; ++u) x[u] = (v.b[u] + off[u]) / diag[u];
                        split_store(a, c, j, k, p0, x);
                    });
    }
}

// sum r^2 over the cells of colour c, r = b - A x, into *out.  The 2 V terms of two
// planes are summed in the element type, everything after them in FP64 (the 256^3 FP32
// step 2.204 ms; with an FP64 addition at each plane 2.216, with none before the warp 2.196).
template <typename T, bool WALLS>
__global__ void __launch_bounds__(128) split_norm_kernel(const SplitArgs<T> a, int c, int chunk,
                                                         double* out) {
    griddep_wait();
    if (griddep_many_blocks()) griddep_launch_dependents();
    constexpr int V = VecOf<T>::V;
    double t = 0.0;
    T sum = T(0);
    int p0, j;
    if (split_column(a, p0, j)) {
        const int k0 = blockIdx.y * chunk, k1 = min(k0 + chunk, a.n[2]);
        split_march<WALLS, true>(a, c, p0, j, k0, k1,
                    [&](int k, const SplitRow<T>& v, const T (&diag)[V], const T (&off)[V]) {
                        const int cnt = row_cells(a, v.s);
#pragma unroll
                        for (int u = 0; u < V; ++u) {
                            const T r = v.b[u] - (diag[u] * v.x[u] - off[u]);
                            if (p0 + u < cnt) sum = fma(r, r, sum);
                        }
                        if ((k & 1) || k + 1 == k1) {
                            t += sum;
                            sum = T(0);
                        }
                    });
    }
    __shared__ double red[4];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        t = red[0] + red[1] + red[2] + red[3];
        if (t != 0.0) atomicAdd(out, t);
    }
}

// The repeated first entry of a row that ends inside a vector: cell i at index
// q of a level by colour.  (With walls and n0 odd the entry is a cell's; there
// the callers store zeros only, in all of x.)
template <typename T>
__device__ __forceinline__ void wrap_entry(const CellArray<T>& c, int i, int q, T v) {
    if (i < 2 && c.stride > (c.n0 >> 1)) c.a[q + (c.n0 >> 1)] = v;
}

// The residual's mean over each coarse cell's children, into the coarse b,
// and a zero coarse x.  After a half-sweep of colour 1 the residual is
// that of the colour-0 children: with x coarsened, child p = I of every row
// (j, k) the cell covers.  A thread takes V coarse cells of a row.
template <typename T, bool WALLS>
__global__ void __launch_bounds__(128) split_restrict_kernel(const SplitArgs<T> a, CellArray<T> cb,
                                                             CellArray<T> cx, int h1, int h2) {
    griddep_wait();
    if (griddep_many_blocks()) griddep_launch_dependents();
    constexpr int V = VecOf<T>::V;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int J = t / a.groups, p0 = (t - J * a.groups) * V, K = blockIdx.y;
    if (J < cb.n1) {
        T sum[V];
#pragma unroll
        for (int u = 0; u < V; ++u) sum[u] = T(0);
        for (int cy = 0; cy < h1; ++cy) {
            const int j = J * h1 + cy;
            split_march<WALLS, true>(a, 0, p0, j, K * h2, (K + 1) * h2,
                               [&](int, const SplitRow<T>& v, const T (&diag)[V], const T (&off)[V]) {
#pragma unroll
                                   for (int u = 0; u < V; ++u)
                                       sum[u] += v.b[u] - (diag[u] * v.x[u] - off[u]);
                               });
        }
#pragma unroll
        for (int u = 0; u < V; ++u)
            if (p0 + u < cb.n0) {
                const int q = cb.index(p0 + u, J, K);
                cb.a[q] = sum[u] / T(2 * h1 * h2);
                cx.a[q] = T(0);
                wrap_entry(cx, p0 + u, q, T(0));
            }
    }
}

// The same with x not coarsened: one coarse cell per thread, its colour-0
// children one by one.
template <typename T, bool WALLS>
__global__ void __launch_bounds__(128) split_restrict_x_kernel(const SplitArgs<T> a,
                                                               CellArray<T> cb, CellArray<T> cx,
                                                               int h1, int h2) {
    griddep_wait();
    if (griddep_many_blocks()) griddep_launch_dependents();
    constexpr int V = VecOf<T>::V;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int J = t / a.n[0], i = t - J * a.n[0], K = blockIdx.y;
    if (J < cb.n1) {
        const int p0 = (i >> 1) / V * V, u0 = (i >> 1) - p0;
        T sum = T(0);
        for (int cz = 0; cz < h2; ++cz)
            for (int cy = 0; cy < h1; ++cy) {
                const int j = J * h1 + cy, k = K * h2 + cz;
                if ((i + j + k) & 1) continue;
                split_march<WALLS, true>(a, 0, p0, j, k, k + 1,
                            [&](int, const SplitRow<T>& v, const T (&diag)[V], const T (&off)[V]) {
#pragma unroll
                                for (int u = 0; u < V; ++u)
                                    if (u == u0) sum += v.b[u] - (diag[u] * v.x[u] - off[u]);
                            });
            }
        const int q = cb.index(i, J, K);
        cb.a[q] = sum / T(h1 * h2);
        cx.a[q] = T(0);
        wrap_entry(cx, i, q, T(0));
    }
}

// x of colour 1 += the correction of its parent cells.  The post-smoothing
// begins with colour 0, which reads colour 1 only, so the old colour 0 needs
// no correction.
template <typename T>
__global__ void __launch_bounds__(128) split_prolong_kernel(const SplitArgs<T> a, CellArray<T> cx,
                                                            int h0, int h1, int h2) {
    griddep_wait();
    if (griddep_many_blocks()) griddep_launch_dependents();
    constexpr int V = VecOf<T>::V;
    int p0, j;
    if (split_column(a, p0, j)) {
        const int k = blockIdx.y, s = (j + k + 1) & 1, cnt = row_cells(a, s);
        const int J = j / h1, K = k / h2;
        T x[V], c[V];
        vload(a.x + a.color + (k * a.n[1] + j) * a.stride + p0, x);
#pragma unroll
        for (int u = 0; u < V; ++u) {
            const int i = 2 * (p0 + u) + s;
            c[u] = p0 + u < cnt ? cx.a[cx.index(h0 == 2 ? i >> 1 : i, J, K)] : T(0);
        }
#pragma unroll
        for (int u = 0; u < V; ++u) x[u] += c[u];
        split_store(a, 1, j, k, p0, x);
    }
}

// The level's x back in mesh order: a vector of each colour per thread makes 2V
// cells of a row (`wide`: rows start on 16 bytes).
template <typename T>
__global__ void __launch_bounds__(128) split_merge_kernel(const SplitArgs<T> a, T* E, bool wide) {
    griddep_wait();
    if (griddep_many_blocks()) griddep_launch_dependents();
    constexpr int V = VecOf<T>::V;
    int p0, j;
    if (!split_column(a, p0, j)) return;
    const int k = blockIdx.y, s0 = (j + k) & 1;        // parity of colour 0
    const int row = (k * a.n[1] + j) * a.stride + p0;
    T e[V], o[V], c[2 * V];
    vload(a.x + (s0 ? a.color : 0) + row, e);          // even cells
    vload(a.x + (s0 ? 0 : a.color) + row, o);
#pragma unroll
    for (int u = 0; u < V; ++u) {
        c[2 * u] = e[u];
        c[2 * u + 1] = o[u];
    }
    T* out = E + (long long)(k * a.n[1] + j) * a.n[0] + 2 * p0;
    if (wide && 2 * (p0 + V) <= a.n[0]) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            typename VecOf<T>::type q;
            q.x = c[h * V];
            q.y = c[h * V + 1];
            if constexpr (V == 4) {
                q.z = c[h * V + 2];
                q.w = c[h * V + 3];
            }
            *reinterpret_cast<typename VecOf<T>::type*>(out + h * V) = q;
        }
    } else {
#pragma unroll
        for (int u = 0; u < 2 * V; ++u)
            if (2 * p0 + u < a.n[0]) out[u] = c[u];
    }
}

// Mean of D over the children, any layout on either side.
template <typename T>
__global__ void __launch_bounds__(128) restrict_any_kernel(CellArray<T> f, CellArray<T> c, bool wrap,
                                                           int h0, int h1, int h2) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int J = t / c.n0, I = t - J * c.n0, K = blockIdx.y;
    if (J >= c.n1) return;
    const T inv = T(1) / T(h0 * h1 * h2);
    T s = T(0);
    for (int cz = 0; cz < h2; ++cz)
        for (int cy = 0; cy < h1; ++cy)
            for (int cx = 0; cx < h0; ++cx)
                s += f.a[f.index(I * h0 + cx, J * h1 + cy, K * h2 + cz)];
    const int q = c.index(I, J, K);
    c.a[q] = s * inv;
    if (wrap) wrap_entry(c, I, q, s * inv);
}

}  // namespace
}  // namespace hh
