// Launch interface of the WENO5-Z + HLL stage kernels (weno.cuh), one
// translation unit per element type like the PLM-minmod + HLLC kernels.
#pragma once
#include "launch.h"

namespace hh {

// The marches of the scheme's directional sweeps on 3D meshes (weno_sweep.cuh):
// blocks of WENO_SWEEP_THREADS columns, a chunk of cells of the march axis each.
inline constexpr int WENO_SWEEP_THREADS = 128;
inline long long march_blocks(long long columns) {
    return (columns + WENO_SWEEP_THREADS - 1) / WENO_SWEEP_THREADS;
}
// Cells per chunk of a march over n cells.  The six warm-up cells, of which four
// only enter the window, cost about four.  Blocks of one SM share its issue
// slots (FP32, from the second on) or its FP64 pipe, so an SM takes the time
// of its blocks one after the other, and one block alone twice its share
// (FP32) or 1.2 times (FP64).
inline int march_chunk(long long columns, int n, bool f64) {
    const long long cols = march_blocks(columns);
    return choose_chunk(cols, n, [&](int z, long long) {
        return std::max(span_steps(cols, n, z, 4.0, SMS), (f64 ? 1.2 : 2.0) * (z + 4.0));
    });
}
// Cells per lane of the x sweeps: segments of 62 (two) or 94 (three), whichever covers
// a row in less work; a segment costs about half a cell per lane besides
// (64 cells: one segment of 94 instead of two of 62; 256: three instead of five: WENO
// 256^3, two steps, 3.95 -> 3.80 ms, advection 0.81 -> 0.77 ms a step).
inline int wx_cells(int n) { return 3.5 * ((n + 93) / 94) < 2.5 * ((n + 61) / 62) ? 3 : 2; }
// Tiles of the fused kernel: 128 cells in 1D, 32 x 8 in 2D and 3D, 32-plane
// z chunks.
inline constexpr int WENO_TX1 = 128, WENO_TX2 = 32, WENO_TY2 = 8, WENO_ZC = 32;

// Blocks of the launch that carries a WENO stage's epilogue (rows of the
// totals partial array): the combining z' march of the sweeps, or the fused
// kernel's grid.
inline long long weno_stage_blocks(const MeshDesc& m, bool sweeps, bool f64) {
    if (m.dim == 3 && sweeps) {
        const long long columns = (long long)m.n[0] * m.n[1];
        const int z = march_chunk(columns, m.n[2], f64);
        return march_blocks(columns) * ((m.n[2] + z - 1) / z);
    }
    return (long long)((m.n[0] + (m.dim == 1 ? WENO_TX1 : WENO_TX2) - 1) / (m.dim == 1 ? WENO_TX1 : WENO_TX2)) *
           (m.dim >= 2 ? (m.n[1] + WENO_TY2 - 1) / WENO_TY2 : 1) *
           (m.dim == 3 ? (m.n[2] + WENO_ZC - 1) / WENO_ZC : 1);
}

// One stage of the second scheme on the mesh: on a 3D mesh with c.scratch
// set, three directional sweeps (c.scratch holds the flux difference
// between them, [5][N] elements, aliasing none of the state buffers);
// otherwise the fused kernel.  Every active axis needs at least three cells.
cudaError_t launch_weno_stage_f32(const MeshDesc& m, const StageCall& c, cudaStream_t s);
cudaError_t launch_weno_stage_f64(const MeshDesc& m, const StageCall& c, cudaStream_t s);

// One Heun stage of the radiation energy advection (WENO5-Z states, Rusanov
// flux) with the fluid state U [5][N] held fixed: stage 1 writes
// Eo = Ec + dt L(Ec), stage 2 Eo = E0/2 + (Ec + dt L(Ec))/2 (Eo may alias E0,
// not Ec).  On a 3D mesh with `scratch` set (N elements aliasing none of the
// other buffers) it runs as three directional sweeps, otherwise as the fused
// kernel.  Every active axis needs at least three cells.
cudaError_t launch_advect_E_stage_f32(const MeshDesc& m, int stage, const void* U, const void* E0,
                                      const void* Ec, void* Eo, double dt, void* scratch,
                                      cudaStream_t s);
cudaError_t launch_advect_E_stage_f64(const MeshDesc& m, int stage, const void* U, const void* E0,
                                      const void* Ec, void* Eo, double dt, void* scratch,
                                      cudaStream_t s);

// The scheme of a handle (hard_hydro.cu): HARD_SCHEME_PLM_HLLC or
// HARD_SCHEME_WENO5Z_HLL.
int handle_scheme(const hard_hydro_s* h);

}  // namespace hh
