// Internal launch interface between the C ABI (hard_hydro.cu) and the kernel
// translation units (one per element type, so that the FP64 one can be built
// without FMA contraction).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

namespace hh {

struct TileDesc {
    int tx, ty, zc;        // tile extents along kernel x', y' and the z chunk
};

// Mesh as the kernels see it: the active axes become kernel axes x', y', z'.
struct MeshDesc {
    int dim;               // number of active axes (0..3)
    int px, py;            // physical axis of kernel x', y'
    int n[3];              // kernel-axis extents (inactive: 1)
    int bc_lo[3], bc_hi[3];
    double dxk[3];         // cell width per kernel axis
    double dx[3];          // cell width per physical axis
    bool act[3];           // physical axis active
    double gamma;
    long long N;           // total cells
    TileDesc auto3[3] = {{32, 8, 32}, {32, 8, 32}, {32, 8, 32}};   // 3D: choose_tile3 by Rule3
};

// ---- chunk lengths by a schedule model ----
// A kernel that marches an axis of n cells in chunks of z has one block per
// tile column and chunk; a block takes (z + over) steps, over standing for its
// warm-up cells, first loads and reductions.  span_steps is the time, in
// steps, until `slots` resident blocks have worked off the whole chunks and
// then the columns' shorter last ones, in launch order.
inline constexpr int SMS = 152;
inline double span_steps(long long cols, int n, int z, double over, long long slots) {
    const long long full = cols * (n / z), q = full / slots, r = full % slots;
    const int rem = n % z;
    const double a = z + over, b = rem + over;
    const double t0 = q * a, t1 = t0 + a;              // slots - r are free at t0, r at t1
    double t = r ? t1 : t0;
    if (!rem) return t;
    if (cols > 64 * slots) return (full * a + cols * b) / slots + 0.5 * a;
    for (int k = 1;; ++k) {                            // the short chunks fill up behind
        const double e0 = t0 + k * b, e1 = t1 + k * b;
        const auto done = [&](double e) {
            long long d = 0;
            if (e >= t0) d += (slots - r) * (long long)((e - t0) / b + 1e-9);
            if (e >= t1) d += r * (long long)((e - t1) / b + 1e-9);
            return d;
        };
        if (done(e0) >= cols) return e0 > t ? e0 : t;
        if (r && done(e1) >= cols && done(t0 + (k + 1) * b) >= cols)
            return e1 < t0 + (k + 1) * b ? e1 : t0 + (k + 1) * b;
    }
}
// The chunk length of the least time(z, blocks).  Lengths that cut n evenly, at
// most 72 (neighbouring columns drift apart in longer ones and lose halo planes
// in L2: 512^3, 2.94 ms a stage with 64 planes, 2.97 with 128) but 512 chunks
// at most; *best (if given) its time.
template <class Time>
inline int choose_chunk(long long cols, int n, const Time& time, double* best = nullptr) {
    double tb = 1e300;
    int zb = n, last = 0;
    for (int c = std::min((n + 71) / 72, 512); c <= n && c <= 512; ++c) {
        const int z = (n + c - 1) / c;
        if (z == last) continue;
        last = z;
        const double t = time(z, cols * ((n + z - 1) / z));
        if (t < tb) {
            tb = t;
            zb = z;
        }
    }
    if (best) *best = tb;
    return zb;
}
// Tile and z chunk of the 3D stage kernels, of 32-wide tiles.  A form's time is
// `first` + the span of its blocks at step[k - 1] a plane where k blocks share an SM,
// `over` planes of each block standing for its warm-up and fixed cost.  Steps measured
// (us): FP32 (warp-specialised, bound by issue) 1.53 a plane of 32 x 8 alone on its
// SM, 1.85 with a second block, 1.67 of 32 x 16 (one block per SM), a block's fixed
// cost ~3 planes; FP64 (bound by its pipe, whatever is resident) 54.6 of 32 x 8
// and 35.1 of 32 x 4 (58 as one of two), fixed cost ~1 plane.  The plain FP32
// kernel fills an SM best with five blocks of 4 rows (512^3: 6.6 ms a stage, 7.9 by
// 8 rows, 8.4 by 16), and blocks of a last wave that leave a fifth of the SMs' places
// free take the step of fewer on an SM.  One fixed 32 x 8 x 32 tile leaves most of
// the chip idle on small meshes (64^3: 54 us a stage, 15 by the rule; plain 104
// and 21) and most of the last wave on others.
enum Rule3 { RULE_FUSED32, RULE_F64, RULE_PLAIN32, RULES3 };
inline TileDesc choose_tile3(const int n[3], Rule3 rule) {
    struct Form { int ty, kmax; double first, over, step[5]; };
    static constexpr Form F32[] = {{16, 1, 0, 3.2, {1.67}}, {8, 2, 0, 3.0, {1.53, 1.85}}};
    static constexpr Form F64[] = {{8, 1, 0, 1.0, {54.6}}, {4, 2, 0, 1.2, {35.1, 58.0}}};
    static constexpr Form PLAIN[] = {{8, 2, 2.1, 0.7, {3.26, 4.34}}, {4, 5, 1.0, 0.8, {3.0, 3.6, 4.0, 4.35, 4.65}}};
    const Form* forms = rule == RULE_F64 ? F64 : rule == RULE_PLAIN32 ? PLAIN : F32;
    const auto columns = [&](int ty) { return (n[0] + 31) / 32 * (long long)((n[1] + ty - 1) / ty); };
    TileDesc td{32, 8, 32};
    double tb = 1e300;
    for (const Form* f = forms; f < forms + 2; ++f) {
        // more rows than a grid of 8-row tiles takes are refused at the launch, as before the rule
        if (n[1] > 8 * 65535 || (n[1] + f->ty - 1) / f->ty > 65535) continue;
        const long long cols = columns(f->ty);
        double t;
        const int z = choose_chunk(cols, n[2], [&](int zc, long long blocks) {
            const int k = (int)std::min<long long>(f->kmax, (blocks + SMS - 1) / SMS);   // blocks on an SM
            const long long slots = (long long)SMS * k, rest = blocks % slots;
            const double s = f->step[k - 1];
            double tz = f->first + span_steps(cols, n[2], zc, f->over, slots) * s;
            const int last = (int)(rest / (SMS * 4 / 5)) + 1;        // on an SM in the last wave
            if (rule == RULE_PLAIN32 && blocks > slots && rest && last < k && n[2] % zc == 0)
                tz -= (zc + f->over) * (s - f->step[last - 1]);
            return tz;
        }, &t);
        if (t < tb) {
            tb = t;
            td = TileDesc{32, f->ty, z};
        }
    }
    // FP32 by TMA in one chunk, as thin meshes are: blocks of other columns come in by
    // and by, which hides more of the fixed cost of the smaller ones.  16 rows
    // (z + 2.4) 1.71 us a wave + 3.3; 8 rows (z + 2.05) 1.74 + 4.4, a last wave of
    // up to 121 blocks at 1.46 (4 planes of 1000^2 163 us a stage against 154, 16 of 500^2
    // 130 against 125, 16 of 256^2 35.5 against 39.0).
    if (rule == RULE_FUSED32 && td.ty == 16 && td.zc == n[2] && n[0] % 4 == 0) {
        const long long b8 = columns(8), b16 = columns(16), rest = b8 % (2 * SMS);
        const double w8 = n[2] + 2.05;
        const double t16 = 3.3 + (n[2] + 2.4) * 1.71 * (double)((b16 + SMS - 1) / SMS);
        const double t8 = 4.4 + w8 * ((double)(b8 / (2 * SMS)) * 1.74 +
                                      (!rest ? 0.0 : rest <= SMS * 4 / 5 ? 1.46 : 1.94));
        if (t8 < t16) td.ty = 8;
    }
    return td;
}

struct StageCall {
    int stage;                     // 1 or 2
    const void* U0;
    const void* Uc;
    void* Uo;
    double dt;                     // used when dt_dev == nullptr
    const double* dt_dev;
    unsigned long long* rate_slot; // nullptr = no rate epilogue
    double* tot_partial;           // nullptr = no totals epilogue
    int* status;
    int zlo = 0, zhi = -1;         // 3D: the kernel-z cells [zlo, zhi) to update (-1: to nz; every
                                   // call takes all of them); zlo a multiple of launch_tile's zc
    const void* zg[2] = {nullptr, nullptr};  // ghost planes of BC_HALO z faces (below, above),
                                             // each [5][2][ny][nx]
    void* scratch = nullptr;       // WENO on 3D meshes: [5][N] flux-difference buffer of the
                                   // sweeps (nullptr: the fused kernel)
};

// Tile configurations per number of active axes (the autotuner's space).
inline constexpr TileDesc TILES3[] = {{32, 8, 32}, {32, 8, 64}, {32, 16, 64}, {64, 8, 64},
                                      {32, 4, 64}, {32, 16, 32}};
// 1D and 2D meshes run one warp per strip of 28 cells (strip.cuh): 32 lanes, ty
// warps per block, zc rows per warp.
inline constexpr TileDesc TILES2[] = {{32, 2, 2}, {32, 2, 4}, {32, 2, 16}};
inline constexpr TileDesc TILES1[] = {{32, 1, 1}, {32, 8, 1}};
inline constexpr int STRIP_CELLS = 28;
// The strips of rows of n0 cells: `full` of them at 32 lanes and, in long walks
// (`share`) where the last cells and their four halo cells leave half a warp and more, one
// whose warps walk `groups` row chunks side by side, `width` lanes each.  Short walks
// are those of meshes that do not fill the chip, whose step is the longest warp's: loads
// from several rows at a time only lengthen it (449 x 42 cells, 20 steps, 218 -> 228 us).
struct StripPlan {
    int full, groups, width;
};
inline __host__ __device__ StripPlan strip_plan(int n0, bool share) {
    const int rest = n0 % STRIP_CELLS, g = 32 / (rest + 4);
    if (!share || rest == 0 || g == 1) return StripPlan{(n0 + STRIP_CELLS - 1) / STRIP_CELLS, 0, 0};
    return StripPlan{n0 / STRIP_CELLS, g, rest + 4};
}
inline bool strip_walks(const TileDesc& t) { return t.zc > 4; }   // rows in a loop, not unrolled
// Warps of a plan over a number of row chunks (I holds the result).
template <typename I>
inline __host__ __device__ I strip_warps(const StripPlan& p, I chunks) {
    return (I)p.full * chunks + (p.groups ? (chunks + (I)p.groups - 1) / (I)p.groups : 0);
}

inline int tile_count(int dim) {
    return dim == 3 ? 6 : dim == 2 ? 3 : dim == 1 ? 2 : 1;
}
inline TileDesc tile_desc(int dim, int tile) {
    if (dim == 3) return TILES3[tile];
    if (dim == 2) return TILES2[tile];
    if (dim == 1) return TILES1[tile];
    return TileDesc{256, 1, 0};
}
// The tile a launch uses: the table's entry, or for tile < 0 the library's
// choice.  2D: rows per warp.  A warp of two rows pays ~1.3x (FP32) / 1.4x
// (FP64) of the work per cell of a long one and of four ~1.15x / 1.2x, for
// more warps and a shorter chain; FP32 hides its latencies with at least 8
// warps per SM, FP64 keeps its pipe busy with 4.  1D: a block per strip for the
// shortest chain and all SMs; once the SMs have five strips each, FP32 meshes take eight
// warps to a block, for an eighth of the atomics on the rate slot and of the rows of
// the totals array (a step of 10^6 cells 31.9 us against 57.8, with totals 68.6
// against 159; of 16000 cells 6.1 against 5.9); FP64 ones, bound by their
// pipe, do not (1168 us against 1108).
inline TileDesc launch_tile(const MeshDesc& m, int kernel, int tile, bool f64) {
    if (tile >= 0) return tile_desc(m.dim, tile);
    if (m.dim == 2) {
        const long long rows = (long long)((m.n[0] + STRIP_CELLS - 1) / STRIP_CELLS) * m.n[1];
        const long long want = 152ll * (f64 ? 4 : 8);
        return TILES2[rows >= 16 * want ? 2 : rows >= 4 * want ? 1 : 0];
    }
    if (m.dim == 1) return TILES1[!f64 && m.n[0] >= STRIP_CELLS * 5 * SMS ? 1 : 0];
    if (m.dim == 3) return m.auto3[f64 ? RULE_F64 : kernel == 0 ? RULE_FUSED32 : RULE_PLAIN32];
    return tile_desc(m.dim, 0);
}
// Blocks the stage kernel launches (rows of the totals partial array).
inline long long stage_blocks(const MeshDesc& m, int kernel, int tile, bool f64) {
    if (m.dim == 0) return 1;
    const TileDesc t = launch_tile(m, kernel, tile, f64);
    if (m.dim < 3) {
        const StripPlan p = strip_plan(m.n[0], strip_walks(t));
        return (strip_warps<long long>(p, (m.n[1] + t.zc - 1) / t.zc) + t.ty - 1) / t.ty;
    }
    const long long gx = (m.n[0] + t.tx - 1) / t.tx;
    const long long gy = (m.n[1] + t.ty - 1) / t.ty;
    const long long gz = (m.n[2] + t.zc - 1) / t.zc;
    return gx * gy * gz;
}

cudaError_t launch_stage_f32(const MeshDesc& m, int kernel, int tile, const StageCall& c,
                             cudaStream_t s);
cudaError_t launch_stage_f64(const MeshDesc& m, int kernel, int tile, const StageCall& c,
                             cudaStream_t s);
// Signal-rate max of U into *rate_slot (which must be zeroed first).
cudaError_t launch_rate_f32(const MeshDesc& m, const void* U, unsigned long long* rate_slot,
                            int* status, cudaStream_t s);
cudaError_t launch_rate_f64(const MeshDesc& m, const void* U, unsigned long long* rate_slot,
                            int* status, cudaStream_t s);
// Per-block partial sums of the 5 fields; returns the number of partial rows.
inline constexpr int TOTALS_BLOCKS = 608;
inline long long totals_blocks() { return TOTALS_BLOCKS; }
cudaError_t launch_totals_f32(const MeshDesc& m, const void* U, double* partial, cudaStream_t s);
cudaError_t launch_totals_f64(const MeshDesc& m, const void* U, double* partial, cudaStream_t s);

// One problem of a batch (see batched.cuh).
struct BatchProblem {
    long long off;        // element offset of the problem's U[5][ny][nx] in the packed buffer
    int nx, ny;           // cells (nz = 1); ny == 1 makes a 1D problem
    int bc;               // boundary kind on all faces
    int pad;
    double gamma;
};

struct BatchCall {
    void* U;
    void* W;
    const BatchProblem* probs;
    const int* order;
    int nprob;
    int nsteps;
    double cfl;
    double* t;
    int* counter;
    int* status;
};

// Batched tile configurations: warps per block.
inline constexpr int BATCH_WARPS[] = {8, 4, 16};
inline constexpr int BATCH_TILE_COUNT = 3;

cudaError_t launch_batched_f32(const BatchCall& c, int tile, cudaStream_t s);
cudaError_t launch_batched_f64(const BatchCall& c, int tile, cudaStream_t s);

// VJP of one stage (adjoint.cuh): gW, 8 slots per cell holding zeros on
// entry, is the primitive cotangent accumulator (cleared again on exit when
// clear_gW);
// out_c (=|+=) b G + J^T(lam G) term; out0 = a G when not null; d/dgamma
// added to *g_gamma.
struct AdjointCall {
    const void* Uc;
    const void* G;
    void* gW;
    void* out_c;
    bool accumulate;
    void* out0;
    double b, a, lam;
    double* g_gamma;
    bool clear_gW;
    int passes = 3;                                // bit 0: the face pass, bit 1: the cell pass
    const void* zg[2] = {nullptr, nullptr};        // BC_HALO z faces: ghost planes of Uc
    void* gwg[2] = {nullptr, nullptr};             // and their cotangent accumulators
};
cudaError_t launch_adjoint_stage_f32(const MeshDesc& m, const AdjointCall& c, cudaStream_t s);
cudaError_t launch_adjoint_stage_f64(const MeshDesc& m, const AdjointCall& c, cudaStream_t s);
// A neighbouring slab's ghost accumulator ([2][ny][nx] records) added into
// planes k0, k0+1 of the accumulator gW.
cudaError_t launch_add_ghost_cotangent_f32(const MeshDesc& m, void* gW, const void* from, int k0,
                                           cudaStream_t s);
cudaError_t launch_add_ghost_cotangent_f64(const MeshDesc& m, void* gW, const void* from, int k0,
                                           cudaStream_t s);

// Read-only view of a handle (hard_hydro.cu); false for a NULL handle.
}  // namespace hh
struct hard_hydro_s;
namespace hh {
bool handle_view(hard_hydro_s* h, const MeshDesc** mesh, int* dtype, int* kernel, int* tile);

// Shared helpers (hard_hydro.cu).
cudaError_t launch_finalize_dt(unsigned long long* rate_slot, double cfl, double t_end,
                               double* t_dev, double* dt_dev, double* dt_log, int step,
                               int* status, cudaStream_t s);
cudaError_t launch_finalize_totals(const double* partial, long long rows, double dV,
                                   double* out5, cudaStream_t s);

}  // namespace hh
