// The interacting pairs of a cell's atoms, found by one warp: the walk that the
// energy, the virial and the FP64 forces of molecular dynamics share.
//
// Of an atom's ~160 candidates one in fifteen interacts, and the FP64 pipe (2
// operations per SM and cycle) takes as long for a few active lanes as for all
// 32.  So the warp holds up to 192 neighbourhood records in registers (six per
// lane, fetched at once; the 27 cells lie end to end, found by a search in their
// offsets), compares each own atom with all of them in FP32, and queues the hits
// in candidate order in a ring in shared memory; the caller evaluates them 32 at
// a time, on full warps.  (One thread per atom, with a list of hits per thread
// and the lists pooled for evaluation, took 145 us for the energy of 192000 atoms
// and 686 for 823000 in 256 replicas, against 133 and 505: its 27 cells are up to
// 18 runs of records that end at different places in every lane.)
//
// A candidate is a hit when it is bonded or closer than its type pair's cutoff,
// with a margin of 2e-5 on FP32's r^2 (good to 9 units of 2^-24): what is left
// out contributes exactly 0.
#pragma once

#include "flipmc_device.cuh"

namespace flipmc {

constexpr int kWalkRecs = 6;       // neighbourhood records per lane
constexpr int kWalkRing = 256;     // queued pairs per warp: 31 waiting and one own atom's 192

struct WalkSmem {
    int4 ring[kWalkRing];          // {dx, dy, dz} = partner - own, tag: type pair | bonded << 4
    int off[28];                   // first candidate of each neighbour cell
    int start[28];                 // its first record
};

__device__ __forceinline__ int walk_types(int tag) { return tag & 15; }
__device__ __forceinline__ bool walk_bonded(int tag) { return (tag & 16) != 0; }

// r^2 of a queued pair in FP64: the integer square is exact, h^2 comes in two
// parts, so it is good to about one unit
struct Quantum2 {
    double hi, lo;
};
__device__ __forceinline__ Quantum2 quantum2(double h)
{
    const double hi = h * h;
    return {hi, fma(h, h, -hi)};
}
__device__ __forceinline__ double walk_r2(const int4 &e, const Quantum2 &q)
{
    const unsigned long long D = (unsigned long long)((long long)e.x * e.x) + (unsigned long long)((long long)e.y * e.y) +
                                 (unsigned long long)((long long)e.z * e.z);
    const double x = __ull2double_rn(D);
    return fma(x, q.hi, x * q.lo);
}

// 1 / x to about one unit: an FP32 reciprocal (2^-21) and one third-order
// Newton step (the error's cube is 2^-63): three FP64 operations one after the
// other, 64 cycles each here, where a division takes 564.  Outside FP32's range,
// the division.
__device__ __forceinline__ double walk_rcp(double x)
{
    const float f = (float)x;
    if (!(fabsf(f) > 1e-30f && fabsf(f) < 1e30f)) return __ddiv_rn(1.0, x);
    const double y = (double)__fdividef(1.0f, f);
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// Pairs of cell c's atoms with the atoms of its neighbourhood (HALF: those of a
// larger site index, so that a walk over all cells meets each pair once).  SLICED:
// of the cell's atoms in groups of 32, number `slice` and every n_slices-th after it.
// The ring holds positions head .. tail - 1, fewer than 32 between calls of P:
// P: own(i0, ni, rec)   the next (at most 32) own atoms; lane i holds atom i's record
//    atom(i, tail)      own atom i's pairs begin at this position
//    eval(at, 32)       evaluate the pairs at positions at, at + 1, ... (whole warp)
//    part(head, tail)   no more pairs of these atoms with this part of the candidates
//    done()             these own atoms are finished
template <bool HALF, bool SLICED, class P>
__device__ __forceinline__ void walk_cell(const DevState &d, const RepInfo &ri, const ModelDev &md, const int4 *rec, int c,
                                          int lane, WalkSmem &sm, int &head, int &tail, P &p, int slice = 0, int n_slices = 1)
{
    constexpr unsigned FULL_WARP = 0xffffffffu;
    const int s0 = d.cell_start[c], n = d.cell_start[c + 1] - s0;
    if (n <= (SLICED ? 32 * slice : 0)) return;
    const int nc = ri.nc, cl = c - ri.cell_off;
    const int cx = cl % nc, cy = (cl / nc) % nc, cz = cl / (nc * nc);
    const bool small = nc == 2;
    const int ns = small ? 8 : 27;
    int cst = 0, cnt = 0;
    if (lane < ns) {
        int ox, oy, oz;
        if (small) {
            ox = lane & 1; oy = (lane >> 1) & 1; oz = lane >> 2;
        } else {
            ox = lane % 3 - 1; oy = (lane / 3) % 3 - 1; oz = lane / 9 - 1;
        }
        const int nb = ri.cell_off + (((cz + oz + nc) % nc) * nc + (cy + oy + nc) % nc) * nc + (cx + ox + nc) % nc;
        cst = d.cell_start[nb];
        cnt = d.cell_start[nb + 1] - cst;
    }
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL_WARP, incl, o);
        if (lane >= o) incl += y;
    }
    __syncwarp();
    if (lane < ns) {
        sm.off[lane] = incl - cnt;
        sm.start[lane] = cst;
    }
    const int K = __shfl_sync(FULL_WARP, incl, 31);
    __syncwarp();
    // cutoffs of the nine type pairs in fixed-point units squared, one per lane
    const float cut = lane < 9 ? md.rc2f[lane] * 1.00002f / ri.hf / ri.hf : 0.f;
    const unsigned lt = (1u << lane) - 1u;
    for (int i0 = SLICED ? 32 * slice : 0; i0 < n; i0 += SLICED ? 32 * n_slices : 32) {
        const int ni = min(32, n - i0);
        const int4 own = rec[s0 + i0 + min(lane, ni - 1)];
        p.own(i0, ni, own);
        for (int c0 = 0; c0 < K; c0 += 32 * kWalkRecs) {
            int4 r[kWalkRecs];
#pragma unroll
            for (int s = 0; s < kWalkRecs; ++s) {
                const int at = c0 + 32 * s + lane;
                r[s] = make_int4(0, 0, 0, kPadWord);
                if (at < K) {
                    int k = 0;
#pragma unroll
                    for (int h = 16; h > 0; h >>= 1)
                        if (k + h < ns && sm.off[k + h] <= at) k += h;
                    r[s] = rec[sm.start[k] + at - sm.off[k]];
                }
            }
            for (int i = 0; i < ni; ++i) {
                const uint32_t mx = (uint32_t)__shfl_sync(FULL_WARP, own.x, i), my = (uint32_t)__shfl_sync(FULL_WARP, own.y, i),
                               mz = (uint32_t)__shfl_sync(FULL_WARP, own.z, i);
                const int mw = __shfl_sync(FULL_WARP, own.w, i);
                const int t3 = 3 * rec_type(mw);
                const float c_a = __shfl_sync(FULL_WARP, cut, t3), c_b = __shfl_sync(FULL_WARP, cut, t3 + 1),
                            c_c = __shfl_sync(FULL_WARP, cut, t3 + 2);
                p.atom(i, tail);
#pragma unroll
                for (int s = 0; s < kWalkRecs; ++s) {
                    if (c0 + 32 * s < K) {
                        const int dx = (int)((uint32_t)r[s].x - mx), dy = (int)((uint32_t)r[s].y - my),
                                  dz = (int)((uint32_t)r[s].z - mz);
                        const float fx = (float)dx, fy = (float)dy, fz = (float)dz;
                        const int tj = rec_type(r[s].w);
                        const uint32_t x = (uint32_t)(r[s].w ^ mw);   // below 16: the same molecule, below 4: the atom
                        const bool near = fmaf(fx, fx, fmaf(fy, fy, fz * fz)) <= (tj == 0 ? c_a : (tj == 1 ? c_b : c_c));
                        // (the words order like the sites: molecule, then slot)
                        const bool other = HALF ? (uint32_t)r[s].w >> 2 > (uint32_t)mw >> 2 : x >= 4u;
                        const bool hit = (near | (x < 16u)) & other & (r[s].w != kPadWord);
                        const unsigned b = __ballot_sync(FULL_WARP, hit);
                        if (hit)
                            sm.ring[(tail + __popc(b & lt)) & (kWalkRing - 1)] =
                                make_int4(dx, dy, dz, (t3 + tj) | (x < 16u ? 16 : 0));
                        tail += __popc(b);
                    }
                }
                __syncwarp();
                for (; tail - head >= 32; head += 32) p.eval(head, 32);
                __syncwarp();
            }
            p.part(head, tail);
        }
        p.done();
    }
}

// The cells of one warp of an energy walk: enough atoms to fill its batches of
// 32 pairs (an atom has about 4 with a larger index and one bond), by the atoms
// per cell of the replica alone, so that a replica's sum is the same in a batch;
// a divisor of 8, as every replica has a multiple of 8 cells.
__host__ __device__ constexpr int walk_cells(int n_sites, int n_cells)
{
    return n_sites >= 14 * n_cells ? 1 : (n_sites >= 8 * n_cells ? 2 : 4);
}

}  // namespace flipmc
