// Molecular dynamics of the same model (Sec. II.D): velocity Verlet with a
// Nose-Hoover thermostat, on the fixed-point positions of the MC state.
#pragma once

#include <cuda_runtime.h>

#include "flipmc_types.h"

namespace flipmc {

// Device state of an MD run: velocities and forces per site (site order),
// thermostat variables per replica.
struct MdDev {
    double *v;         // 3 per site
    double *F;         // 3 per site
    double *xi;        // per replica: thermostat friction at the end of the last step
    double *eta;       // per replica: its time integral (for the conserved energy)
    double *xi_mid;    // per replica: both after the first thermostat half step of the next step,
    double *eta_mid;   //              which follows from the same kinetic energy
    double *scale;     // per replica: exp(-xi_mid dt/2)
    const double *T;   // per replica: bath temperature
    const double *Q;   // per replica: thermostat mass g T tau^2, g = 3 N
    Units units;       // blocks of the force kernel: kMdWarps of a replica's warps (FP64; md_warps), or 32 records (FP32)
    double *part;      // per block: partial sum of v^2
    unsigned *arrived; // per replica: blocks that have written theirs (zero between steps)
    int fp32_forces;   // 1: pair forces in FP32 (velocities, positions and thermostat stay FP64)
    double dt;
    double hdt;        // dt / 2
};

// The warps of the FP64 forces of a replica: one per cell; where most cells are
// empty and there are many, one for `cells` neighbouring cells; where cells are
// crowded, `slices` for each, which share out its atoms in groups of 32.
// With a warp per cell a dilute system had little but the ends of the step to its
// blocks, all of them at one counter (8000 molecules at a density of 0.05, 4.6 cells
// per atom: 229 us a step, now 117; at 0.02, 12 cells per atom: 470, now 136), and
// crowded cells had too few warps (1000 molecules in eight cells 11955, now 8670, nearly
// all of it the ordering of the cells).  About an atom to a warp is little enough to
// wait for, and 4096 warps fill the GPU: 216 molecules at 0.05, in 2744 cells, take
// 25 with a warp per cell and 33 with one for four cells.
struct MdWarps {
    int cells, slices, n;
};
__host__ __device__ inline MdWarps md_warps(int n_sites, int n_cells)
{
    const int per_atom = n_cells / n_sites, spare = n_cells / 4096, per_cell = n_sites / n_cells;
    const int c = per_atom < spare ? per_atom : spare;
    MdWarps w;
    w.cells = c < 1 ? 1 : (c < 16 ? c : 16);
    w.slices = per_cell <= 32 ? 1 : (per_cell + 31) / 32;
    w.n = w.slices > 1 ? w.slices * n_cells : (n_cells + w.cells - 1) / w.cells;
    return w;
}

// The forces of the current state and the first thermostat half step of the first step.
void launch_md_setup(const DevState &d, int buf, const MdDev &m, cudaStream_t st);
// The forces alone (the velocities and the thermostat go on as they are).
void launch_md_forces(const DevState &d, int buf, const MdDev &m, cudaStream_t st);
// One step from the cell-sorted records of buf into buf ^ 1.  cell_count must be zero, and is again afterwards.
void launch_md_step(const DevState &d, int buf, const MdDev &m, cudaStream_t st);

}  // namespace flipmc
