// Energy and time-correlation kernels.
#pragma once

#include <cuda_runtime.h>

#include "flipmc_types.h"

namespace flipmc {

// Time origin of the correlation functions (Sec. III.B).
struct ObsState {
    long long *X0;   // 3 per site: unwrapped fixed point at t0
    int *kref;       // per molecule: slot of the atom that was type B at t0
    double *u0;      // 3 per molecule: unit orientation at t0
};

// A wavevector of one replica in turns per quantum (turns.cuh): per axis the
// 96-bit fraction of kappa = q h / 2 pi (k2 the highest word), and the phase of
// the displacement 2^31 on every axis (the kernels add 2^31 to a displacement
// to make it unsigned).
struct alignas(16) Turns {
    uint32_t k0[3], k1[3], k2[3];
    uint32_t bad;    // a component is not finite: every result is NaN
    uint64_t bias;
};
// out[r * n_q + k] = the wavevector qv[3 k ..] of every replica; over_three:
// divided by three (for sums of three displacements, a molecule's atoms)
void launch_turns(const DevState &d, const double *qv, int n_q, bool over_three, Turns *out, cudaStream_t st);

// FP64 energy per replica into e_out_dev[n_rep]; part: one double per block (d.cells.n).
void launch_energy(const DevState &d, int buf, double *part, double *e_out_dev, cudaStream_t st);
// Periodic drift check: drift[2r] = |e_run - E| / |E| (last), drift[2r+1] its
// largest value; one recompute counted; e_run restarts from E[r].
void launch_drift(const DevState &d, const double *E, double *drift, cudaStream_t st);
// S(q) per (replica, wavevector) of the records of buf: out[r * stride + k] =
// |sum_i exp(i q_k . x_i)|^2 / N for the n_q wavevectors of turns; part:
// sq_parts(max_sites) * n_q * n_rep pairs of doubles.
int sq_parts(int max_sites);
void launch_sq(const DevState &d, int buf, const Turns *turns, int n_q, int max_sites, double2 *part, double *out,
               int stride, cudaStream_t st);
// Pair-distance counts per replica and bin (every pair once) of the records of buf; counts zeroed by the caller.
void launch_pair_hist(const DevState &d, int buf, int max_sites, double dr, int n_bins, unsigned long long *counts,
                      cudaStream_t st);
// FP64 pair virial sum W = sum_{i<j} -r dphi/dr per replica into w_out_dev[n_rep].
void launch_virial(const DevState &d, int buf, double *part, double *w_out_dev, cudaStream_t st);
// unwrapped positions (3 per site) and types in site order
void launch_gather(const DevState &d, int buf, long long *X, int *types, cudaStream_t st);
void launch_set_t0(const DevState &d, const long long *X, const int *types, const ObsState &o, cudaStream_t st);

// The molecules of every replica in chunks of at most kCorrChunk, none
// spanning two replicas (one block of the correlation kernels each).
struct MolChunks {
    const int *m0;           // per chunk: first molecule (global index), m0[n] = total molecules
    const int *rep0;         // per replica: first chunk; [n_rep] = n
    int n;
};
constexpr int kCorrChunk = 32;   // molecules per block: one per lane

// Per particle F_s (fs_site), F_s^cm and C_2 (per molecule) and, per replica,
// out[3 r + {0,1,2}] = their means; part: kCorrPart doubles per chunk.
void launch_observables(const DevState &d, const long long *X, const ObsState &o, const MolChunks &mc, const Turns *ta,
                        int nqa, const Turns *tc, int nqc, double *fs_site, double *fscm_mol, double *c2_mol,
                        double *part, double *out, cudaStream_t st);

// Multiple-origin correlations: the origins live in slots; each slot holds an
// ObsState's arrays (slot s at X0 + 3 N s, kref + M s, u0 + 3 M s).
struct CorrDev {
    const long long *X0;
    const int *kref;
    const double *u0;
    size_t n_sites;             // all replicas
    const Turns *ta;            // n_qa wavevectors (atoms) per replica
    const Turns *tc;            // n_qc wavevectors (centres of mass) per replica
    int n_qa, n_qc;
    MolChunks chunks;
    double *partials;           // kCorrPart per (pair, chunk)
    double *acc;                // MC_CORR_NSUM per (replica, lag)
    int n_lags;
};

constexpr int kCorrMaxPairs = 32;       // (origin, lag) pairs per launch
constexpr int kCorrPart = 8;            // partial sums per (pair, chunk)

// The (origin slot, lag index) pairs measured at one time.
struct CorrPairs {
    int n;
    int slot[kCorrMaxPairs];
    int lag[kCorrMaxPairs];
};

// Per-particle correlations of each pair against the current unwrapped
// positions X, summed per replica into the accumulators (fixed order).
void launch_corr_sample(const DevState &d, const long long *X, const CorrDev &c, const CorrPairs &p, cudaStream_t st);

}  // namespace flipmc
