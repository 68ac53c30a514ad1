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
    Units units;       // blocks of the force kernel: kMdWarps cells (FP64), or 32 records (FP32)
    double *part;      // per block: partial sum of v^2
    unsigned *arrived; // per replica: blocks that have written theirs (zero between steps)
    int fp32_forces;   // 1: pair forces in FP32 (velocities, positions and thermostat stay FP64)
    double dt;
    double hdt;        // dt / 2
};

// The forces of the current state and the first thermostat half step of the first step.
void launch_md_setup(const DevState &d, int buf, const MdDev &m, cudaStream_t st);
// One step from the cell-sorted records of buf into buf ^ 1.  cell_count must be zero, and is again afterwards.
void launch_md_step(const DevState &d, int buf, const MdDev &m, cudaStream_t st);

}  // namespace flipmc
