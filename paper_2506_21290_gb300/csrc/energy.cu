// Total energy (Eq. 1 + Eq. 2, FP64) over the cell neighbourhoods, and the
// time correlations of Sec. III.B (Eq. 5-7).
#include <algorithm>

#include "cell_list.h"
#include "energy.h"
#include "flipmc_device.cuh"
#include "pair_walk.cuh"
#include "turns.cuh"

namespace flipmc {

// ln y to about two units, y in (0, 1]: the atanh series of ln_series with
// fused steps and the walk's reciprocal.  NaN below 0, -inf at 0.
__device__ __forceinline__ double walk_ln(double y)
{
    const long long bits = __double_as_longlong(y);
    int e = (int)((bits >> 52) & 0x7FF) - 1023;
    double m = __longlong_as_double((bits & 0x000FFFFFFFFFFFFFll) | 0x3FF0000000000000ll);
    if (m > 0x1.6a09e667f3bcdp+0) {
        m *= 0.5;
        e += 1;
    }
    const double z = (m - 1.0) * walk_rcp(m + 1.0), w = z * z;
    double s = 2.0 / 23.0;
    s = fma(s, w, 2.0 / 21.0);
    s = fma(s, w, 2.0 / 19.0);
    s = fma(s, w, 2.0 / 17.0);
    s = fma(s, w, 2.0 / 15.0);
    s = fma(s, w, 2.0 / 13.0);
    s = fma(s, w, 2.0 / 11.0);
    s = fma(s, w, 2.0 / 9.0);
    s = fma(s, w, 2.0 / 7.0);
    s = fma(s, w, 2.0 / 5.0);
    s = fma(s, w, 2.0 / 3.0);
    s = fma(s, w, 2.0);
    const double r = fma((double)e, 0x1.62e42fefa39efp-1, z * s);
    return y > 0.0 ? r : (y == 0.0 ? -__longlong_as_double(0x7FF0000000000000ll) : __longlong_as_double(0x7FF8000000000000ll));
}

// Energy (VIRIAL = false) or pair virial (VIRIAL = true) of every replica: each
// pair from its atom of the smaller site index (pair_walk.cuh), FP64.  A warp
// walks one to four cells and keeps what does not fill a batch of 32 pairs for
// the next; bonds, whose Eq. 2 costs three times Eq. 1, wait in a ring of their
// own for full batches.  The sums (per lane, then lanes, warps and, in a second
// kernel, blocks) run in a fixed order: the same on every run for a given state.
// (No counter tells a last block to add the blocks' sums: mc_energy_device is
// asynchronous, so two of these may overlap on two streams, or in two replayed
// graphs, with one handle's workspace.  Both write the same numbers to it.)
// Energy of 24000 atoms 42 us (62 when every lane of a warp walked a neighbour
// cell and bonds shared the batches), of 192000 atoms 124 (290), of 256 replicas
// with 823000 atoms 494 (1161), both kernels.  96 registers with 52 bytes of
// spills: without them at 116 registers the last two take 133 and 559, and at 92
// registers 122 and 496.
template <bool VIRIAL>
struct EnergyWalk {
    const ModelDev &md;
    const Quantum2 hh;
    const double c24;
    const int4 *ring;
    double *bond_r2;               // [64] waiting bonds, and their type pairs
    int *bond_ab;
    const int lane;
    int bond_head = 0, bond_tail = 0;
    double acc = 0.0;

    __device__ void own(int, int, const int4 &) {}
    __device__ void atom(int, int) {}
    __device__ void part(int, int) {}
    __device__ void done() {}
    __device__ void eval(int at, int n)
    {
        const bool on = lane < n;
        const int4 e = ring[(at + (on ? lane : 0)) & (kWalkRing - 1)];
        const int ab = walk_types(e.w);
        const double r2 = walk_r2(e, hh);
        const double t = md.s2[ab] * walk_rcp(r2);
        const double s6 = t * t * t;
        const double v = VIRIAL ? c24 * (s6 * fma(2.0, s6, -1.0)) : fma(md.e4 * s6, s6 - 1.0, md.eps);
        if (on && r2 < md.rc2[ab]) acc += v;
        const bool bond = on && walk_bonded(e.w);
        const unsigned b = __ballot_sync(0xffffffffu, bond);
        if (bond) {
            const int k = (bond_tail + __popc(b & ((1u << lane) - 1u))) & 63;
            bond_r2[k] = r2;
            bond_ab[k] = ab;
        }
        bond_tail += __popc(b);
        if (bond_tail - bond_head >= 32) bonds(32);
    }
    __device__ void bonds(int n)
    {
        __syncwarp();
        if (lane < n) {
            const int k = (bond_head + lane) & 63;
            const double x = bond_r2[k] * md.invR2[bond_ab[k]];
            acc += VIRIAL ? 2.0 * md.nke * x * walk_rcp(1.0 - x) : md.nke * walk_ln(1.0 - x);
        }
        bond_head += n;
        __syncwarp();
    }
};

template <bool VIRIAL>
__global__ void __launch_bounds__(32 * kEnergyWarps) pair_energy_kernel(DevState d, int buf, double *part)
{
    __shared__ WalkSmem walk[kEnergyWarps];
    __shared__ double bond_r2[kEnergyWarps][64], red[kEnergyWarps];
    __shared__ int bond_ab[kEnergyWarps][64];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int r = 0, c0 = 0;
    if (d.cells.unit != nullptr) {
        const int2 u = d.cells.unit[blockIdx.x];
        r = u.x;
        c0 = u.y;
    }
    const RepInfo ri = d.rep[r];
    const int per = walk_cells(ri.n_sites, ri.nc * ri.nc * ri.nc);
    if (d.cells.unit == nullptr) c0 = blockIdx.x * kEnergyWarps * per;
    const ModelDev &md = *d.model;
    EnergyWalk<VIRIAL> p{md, quantum2(ri.h), 6.0 * md.e4, walk[w].ring, bond_r2[w], bond_ab[w], lane};
    int head = 0, tail = 0;
    for (int k = 0; k < per; ++k)
        walk_cell<true, false>(d, ri, md, d.rec[buf], c0 + w * per + k, lane, walk[w], head, tail, p);
    if (tail > head) p.eval(head, tail - head);
    if (p.bond_tail > p.bond_head) p.bonds(p.bond_tail - p.bond_head);
    double v = p.acc;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (lane == 0) red[w] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < kEnergyWarps; ++k) v = __dadd_rn(v, red[k]);
        part[blockIdx.x] = v;
    }
}

// Sum of each replica's parts (one block each), in a fixed order: thread t adds
// parts t, t + 256, ..., eight loads in flight; then a tree.
constexpr int kPartsThreads = 256;

__global__ void __launch_bounds__(kPartsThreads) replica_parts_kernel(DevState d, const double *part, double *out)
{
    const int r = blockIdx.x, tid = threadIdx.x;
    const int b0 = d.cells.unit != nullptr ? d.cells.rep0[r] : 0;
    const int nb = d.cells.unit != nullptr ? d.cells.rep0[r + 1] - b0 : d.cells.n;
    const double *p = part + b0;
    double s = 0.0;
    for (int k = tid; k < nb; k += 8 * kPartsThreads) {
        double v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = k + j * kPartsThreads < nb ? p[k + j * kPartsThreads] : 0.0;
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (k + j * kPartsThreads < nb) s = __dadd_rn(s, v[j]);
    }
    __shared__ double red[kPartsThreads];
    red[tid] = s;
    __syncthreads();
    if (tid < 64) red[tid] = __dadd_rn(__dadd_rn(red[tid], red[tid + 64]), __dadd_rn(red[tid + 128], red[tid + 192]));
    __syncthreads();
    for (int o = 32; o > 0; o >>= 1) {
        if (tid < o) red[tid] = __dadd_rn(red[tid], red[tid + o]);
        __syncthreads();
    }
    if (tid == 0) out[r] = red[0];
}

template <bool VIRIAL>
static void launch_walk(const DevState &d, int buf, double *part, double *out, cudaStream_t st)
{
    pair_energy_kernel<VIRIAL><<<d.cells.n, 32 * kEnergyWarps, 0, st>>>(d, buf, part);
    replica_parts_kernel<<<d.n_rep, kPartsThreads, 0, st>>>(d, part, out);
}

void launch_energy(const DevState &d, int buf, double *part, double *e_out_dev, cudaStream_t st)
{
    launch_walk<false>(d, buf, part, e_out_dev, st);
}

void launch_virial(const DevState &d, int buf, double *part, double *w_out_dev, cudaStream_t st)
{
    launch_walk<true>(d, buf, part, w_out_dev, st);
}

// Drift check of the running total against a fresh FP64 recompute E, per
// replica (one thread each): the relative drift |e_run - E| / |E| into
// drift[2r] (last) and drift[2r + 1] (largest so far), one more recompute
// counted, and e_run restarted from E.
__global__ void drift_kernel(DevState d, const double *E, double *drift)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= d.n_rep) return;
    const double e = E[r];
    const double rel = fabs(d.e_run[r] - e) / fabs(e);
    drift[2 * r] = rel;
    drift[2 * r + 1] = fmax(drift[2 * r + 1], rel);
    d.stats[(size_t)r * STAT_N + STAT_RECOMP] += 1;
    d.e_run[r] = e;
}

void launch_drift(const DevState &d, const double *E, double *drift, cudaStream_t st)
{
    drift_kernel<<<(d.n_rep + 127) / 128, 128, 0, st>>>(d, E, drift);
}

// Unwrapped fixed-point positions and types in site-index order.
__global__ void gather_kernel(DevState d, int buf, long long *X, int *types)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= d.n_sites) return;
    const int r = d.rep_of_site[g];
    const int off = d.rep[r].site_off;
    const int4 rc = d.rec[buf][g];
    const int s = off + rec_site(rc.w);
    X[3 * s + 0] = (long long)(uint32_t)rc.x + ((long long)d.img[3 * s + 0] << 32);
    X[3 * s + 1] = (long long)(uint32_t)rc.y + ((long long)d.img[3 * s + 1] << 32);
    X[3 * s + 2] = (long long)(uint32_t)rc.z + ((long long)d.img[3 * s + 2] << 32);
    types[s] = rec_type(rc.w);
}

// Orientation of molecule m (global index): centroid -> site kref, from the
// wrapped positions with intramolecular minimum images (equal masses).
__device__ void orientation(const long long *X, int m, int kref, double h, double *u)
{
    const long long *x0 = X + 9 * (size_t)m;
    double rel[3][3];
    for (int k = 0; k < 3; ++k)
        for (int ax = 0; ax < 3; ++ax) rel[k][ax] = (double)(int)((uint32_t)x0[3 * k + ax] - (uint32_t)x0[ax]) * h;
    double n2 = 0.0;
    for (int ax = 0; ax < 3; ++ax) {
        const double cm = ((rel[0][ax] + rel[1][ax]) + rel[2][ax]) / 3.0;
        u[ax] = rel[kref][ax] - cm;
        n2 += u[ax] * u[ax];
    }
    const double inv = 1.0 / sqrt(n2);
    for (int ax = 0; ax < 3; ++ax) u[ax] *= inv;
}

__global__ void set_t0_kernel(DevState d, const long long *X, const int *types, ObsState o)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= d.n_sites / 3) return;
    for (int k = 0; k < 9; ++k) o.X0[9 * (size_t)m + k] = X[9 * (size_t)m + k];
    int kref = 0;
    for (int s = 2; s >= 0; --s)
        if (types[3 * m + s] == 1) kref = s;
    o.kref[m] = kref;
    const int r = d.rep_of_site[3 * m];
    double u[3];
    orientation(X, m, kref, d.rep[r].h, u);
    for (int ax = 0; ax < 3; ++ax) o.u0[3 * (size_t)m + ax] = u[ax];
}

// ---------------------------------------------------------------------------
// Correlations of Eq. 5-7
// ---------------------------------------------------------------------------
// What bounds them: 3 n_qa + n_qc cosines per molecule and origin.  As FP64
// cosines they kept the FP64 pipe 86% busy; with the integer cosines of
// turns.cuh a launch for 8 x 1000 molecules with 48 wavevectors of each kind
// (1 to 2 origins) takes 20.5 us instead of 320 (integer multiplies), and the
// observables of 8000 molecules 17.3 instead of 174.6.
//
// A block takes 32 molecules of one replica.  Their displacements are staged
// once as 32-bit words; lane l of every warp holds molecule l, and the eight
// warps share out the wavevectors, so that a few thousand molecules fill the
// GPU (one molecule per thread left most of it idle) and a wavevector is one
// broadcast load.  The warps' integer sums add up in shared memory, exactly;
// what is left in FP64 (C_2, the squares, the sums over molecules) runs on
// full warps, about 45 operations per 32 molecules.
constexpr int kSlices = 8;
constexpr double kCosUnit = 0x1p53;   // cos_turn's 1

struct RelaxSmem {
    uint32_t lo[12][kCorrChunk];      // per atom and axis, then of the three atoms' sum: displacement + 2^31 ...
    int hi[12][kCorrChunk];           // ... and its multiples of 2^32
    uint32_t q[9][kCorrChunk];        // wrapped positions now
    long long part[kSlices][4][kCorrChunk];
    int bad;
};

// sm.part[w][k][l] = warp w's share of sum_q cos of atom k (k = 3: centre of
// mass) of molecule m0 + l, in units of 2^-53; lanes past nm hold no molecule.
// Leaves the block synchronised.
__device__ __forceinline__ void relax_cosines(RelaxSmem &sm, const long long *X, const long long *X0, int m0, int nm,
                                              const Turns *ta, int nqa, const Turns *tc, int nqc)
{
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    int far = 0;
    for (int i = tid; i < 9 * kCorrChunk; i += 32 * kSlices) {
        const int m = i / 9, c = i - 9 * m;
        long long d = 0;
        uint32_t q = 0;
        if (m < nm) {
            const long long x = X[9 * (size_t)m0 + i];
            d = x - X0[9 * (size_t)m0 + i];
            q = (uint32_t)x;
        }
        d += 1ll << 31;
        sm.q[c][m] = q;
        sm.lo[c][m] = (uint32_t)d;
        sm.hi[c][m] = (int)(d >> 32);
        far |= (int)(d >> 32);
    }
    if (tid == 0) sm.bad = 0;
    __syncthreads();
    if (tid < 3 * kCorrChunk) {
        const int m = lane, ax = w;
        long long d = 1ll << 31;
        for (int k = 0; k < 3; ++k)
            d += ((long long)sm.hi[3 * k + ax][m] << 32) + (long long)sm.lo[3 * k + ax][m] - (1ll << 31);
        sm.lo[9 + ax][m] = (uint32_t)d;
        sm.hi[9 + ax][m] = (int)(d >> 32);
        far |= (int)(d >> 32);
    }
    far = __syncthreads_or(far);
    uint32_t u[12];
#pragma unroll
    for (int c = 0; c < 12; ++c) u[c] = sm.lo[c][lane];
    long long s[4] = {0, 0, 0, 0};
    auto cosine = [&](const Turns &t, int k) {
        uint64_t p = turn_phase(t, u[3 * k], u[3 * k + 1], u[3 * k + 2]) - t.bias;
        if (far) p += turn_phase_boxes(t, sm.hi[3 * k][lane], sm.hi[3 * k + 1][lane], sm.hi[3 * k + 2][lane]);
        return cos_turn(p);
    };
    unsigned bad = 0;
    for (int q = w; q < nqa; q += kSlices) {
        const Turns t = ta[q];
        bad |= t.bad;
#pragma unroll
        for (int k = 0; k < 3; ++k) s[k] += cosine(t, k);
    }
    // (the warps take the centre-of-mass vectors from the other end, so that
    // short lists of both kinds do not meet in the same warps)
    for (int q = kSlices - 1 - w; q < nqc; q += kSlices) {
        const Turns t = tc[q];
        bad |= t.bad << 1;
        s[3] += cosine(t, 3);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) sm.part[w][k][lane] = s[k];
    if (lane == 0 && bad) atomicOr(&sm.bad, (int)bad);
    __syncthreads();
}

// the sum over the wavevectors of quantity k of molecule l, as a double (NaN
// when one of its wavevectors is not finite)
__device__ __forceinline__ double relax_sum(const RelaxSmem &sm, int k, int l)
{
    long long s = 0;
#pragma unroll
    for (int w = 0; w < kSlices; ++w) s += sm.part[w][k][l];
    return (sm.bad >> (k == 3)) & 1 ? __longlong_as_double(0x7FF8000000000000ll) : (double)s;
}

// C_2 of molecule l against its orientation u0 (unit vector): the current
// orientation is along three times (site kref - centroid), an integer vector.
__device__ __forceinline__ double relax_c2(const RelaxSmem &sm, int l, int kref, const double *u0)
{
    double dot = 0.0, n2 = 0.0;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const int a = (int)(sm.q[3 + ax][l] - sm.q[ax][l]), b = (int)(sm.q[6 + ax][l] - sm.q[ax][l]);
        const long long mine = kref == 0 ? 0ll : (kref == 1 ? (long long)a : (long long)b);
        const double v = (double)(3 * mine - a - b);
        dot += v * u0[ax];
        n2 += v * v;
    }
    return 1.5 * (dot * dot / n2) - 0.5;
}

__global__ void __launch_bounds__(32 * kSlices) observables_kernel(DevState d, const long long *X, ObsState o,
                                                                   MolChunks mc, const Turns *ta, int nqa,
                                                                   const Turns *tc, int nqc, double *fs_site,
                                                                   double *fscm_mol, double *c2_mol, double *part)
{
    __shared__ RelaxSmem sm;
    const int m0 = mc.m0[blockIdx.x], nm = mc.m0[blockIdx.x + 1] - m0;
    const int r = d.rep_of_site[3 * m0];
    relax_cosines(sm, X, o.X0, m0, nm, ta + (size_t)r * nqa, nqa, tc + (size_t)r * nqc, nqc);
    // warps 0-2: the atoms, warp 3: the centres of mass, warp 4: the orientations
    const int l = threadIdx.x & 31, k = threadIdx.x >> 5, m = m0 + l;
    if (k > 4) return;
    double v = 0.0;
    if (l < nm) {
        if (k == 4) v = c2_mol[m] = relax_c2(sm, l, o.kref[m], o.u0 + 3 * (size_t)m);
        else if (k == 3) v = fscm_mol[m] = relax_sum(sm, 3, l) / (kCosUnit * nqc);
        else v = fs_site[3 * (size_t)m + k] = relax_sum(sm, k, l) / (kCosUnit * nqa);
    }
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, s));
    if (l == 0) part[(size_t)blockIdx.x * kCorrPart + k] = v;
}

// Means per replica: the chunk sums (thread k takes chunks k, k + 128, ... in
// order, then a fixed tree).
__global__ void __launch_bounds__(128) observables_mean_kernel(DevState d, MolChunks mc, const double *part, double *out)
{
    const int r = blockIdx.x;
    double S[3] = {0.0, 0.0, 0.0};
    for (int k = mc.rep0[r] + threadIdx.x; k < mc.rep0[r + 1]; k += 128) {
        const double *p = part + (size_t)k * kCorrPart;
        S[0] = __dadd_rn(S[0], __dadd_rn(__dadd_rn(p[0], p[1]), p[2]));
        S[1] = __dadd_rn(S[1], p[3]);
        S[2] = __dadd_rn(S[2], p[4]);
    }
    __shared__ double red[3][128];
    for (int j = 0; j < 3; ++j) red[j][threadIdx.x] = S[j];
    __syncthreads();
    for (int w = 64; w > 0; w >>= 1) {
        if (threadIdx.x < w)
            for (int j = 0; j < 3; ++j) red[j][threadIdx.x] = __dadd_rn(red[j][threadIdx.x], red[j][threadIdx.x + w]);
        __syncthreads();
    }
    if (threadIdx.x < 3) {
        const int n = d.rep[r].n_sites;
        out[3 * (size_t)r + threadIdx.x] = red[threadIdx.x][0] / (double)(threadIdx.x == 0 ? n : n / 3);
    }
}

// Block (chunk, pair): the seven sums of the chunk's molecules that the
// statistics need: of F_s of the three atoms, of its squares, of F_s^cm, of its
// square, of C_2, of its square, and of C_2 F_s^cm.
__global__ void __launch_bounds__(32 * kSlices) corr_chunk_kernel(DevState d, const long long *X, CorrDev c, CorrPairs p)
{
    __shared__ RelaxSmem sm;
    const int chunk = blockIdx.x, pr = blockIdx.y;
    const int m0 = c.chunks.m0[chunk], nm = c.chunks.m0[chunk + 1] - m0;
    const int slot = p.slot[pr];
    const size_t M = c.n_sites / 3;
    const int r = d.rep_of_site[3 * m0];
    relax_cosines(sm, X, c.X0 + (size_t)slot * 3 * c.n_sites, m0, nm, c.ta + (size_t)r * c.n_qa, c.n_qa,
                  c.tc + (size_t)r * c.n_qc, c.n_qc);
    if (threadIdx.x >= 32) return;
    const int l = threadIdx.x;
    double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (l < nm) {
        const size_t m = (size_t)slot * M + m0 + l;
        const double c2 = relax_c2(sm, l, c.kref[m], c.u0 + 3 * m);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const double f = relax_sum(sm, k, l);
            v[0] += f;
            v[1] += f * f;
        }
        const double f = relax_sum(sm, 3, l);
        v[2] = f;
        v[3] = f * f;
        v[4] = c2;
        v[5] = c2 * c2;
        v[6] = c2 * f;
    }
    // sum over the lanes in a fixed order, halving the quantities per lane with
    // the lanes (9 additions instead of 35); lane l ends with quantity l >> 2
#pragma unroll
    for (int o = 16, h = 4; o >= 4; o >>= 1, h >>= 1) {
        const bool up = (l & o) != 0;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (i < h) {
                const double give = up ? v[i] : v[i + h], keep = up ? v[i + h] : v[i];
                v[i] = __dadd_rn(keep, __shfl_xor_sync(0xffffffffu, give, o));
            }
    }
    v[0] = __dadd_rn(v[0], __shfl_xor_sync(0xffffffffu, v[0], 2));
    v[0] = __dadd_rn(v[0], __shfl_xor_sync(0xffffffffu, v[0], 1));
    const int j = l >> 2;
    if ((l & 3) == 0 && j < 7) {
        // the cosine sums over wavevectors become means (exact where all are 1)
        const double A = kCosUnit * c.n_qa, C = kCosUnit * c.n_qc;
        const double unit = j == 0 ? A : j == 1 ? A * A : j == 2 || j == 6 ? C : j == 3 ? C * C : 1.0;
        c.partials[((size_t)pr * c.chunks.n + chunk) * kCorrPart + j] = v[0] / unit;
    }
}

// Block (pair, replica): the replica's chunk sums (thread k takes chunks k,
// k + 128, ... in order, then a fixed tree over the threads), then the
// sample's contribution to the replica's accumulators of the pair's lag.
// Different origins never share a lag at one time, so each accumulator has
// one writer per launch.
__global__ void __launch_bounds__(128) corr_finish_kernel(DevState d, CorrDev c, CorrPairs p)
{
    const int pr = blockIdx.x / d.n_rep, r = blockIdx.x - pr * d.n_rep;
    double S[7] = {0, 0, 0, 0, 0, 0, 0};
    for (int k = c.chunks.rep0[r] + threadIdx.x; k < c.chunks.rep0[r + 1]; k += 128)
        for (int j = 0; j < 7; ++j) S[j] = __dadd_rn(S[j], c.partials[((size_t)pr * c.chunks.n + k) * kCorrPart + j]);
    __shared__ double red[7][128];
    for (int j = 0; j < 7; ++j) red[j][threadIdx.x] = S[j];
    __syncthreads();
    for (int w = 64; w > 0; w >>= 1) {
        if (threadIdx.x < w)
            for (int j = 0; j < 7; ++j) red[j][threadIdx.x] = __dadd_rn(red[j][threadIdx.x], red[j][threadIdx.x + w]);
        __syncthreads();
    }
    if (threadIdx.x != 0) return;
    for (int j = 0; j < 7; ++j) S[j] = red[j][0];
    const double M = (double)(d.rep[r].n_sites / 3), N = 3.0 * M;
    const double fs = S[0] / N, fcm = S[2] / M, c2 = S[4] / M;
    double *a = c.acc + ((size_t)r * c.n_lags + p.lag[pr]) * MC_CORR_NSUM;
    a[0] += 1.0;
    a[1] += fs;
    a[2] += fs * fs;
    a[3] += S[0];
    a[4] += S[1];
    a[5] += fcm;
    a[6] += fcm * fcm;
    a[7] += S[2];
    a[8] += S[3];
    a[9] += c2;
    a[10] += c2 * c2;
    a[11] += S[4];
    a[12] += S[5];
    a[13] += S[6];
}

void launch_corr_sample(const DevState &d, const long long *X, const CorrDev &c, const CorrPairs &p, cudaStream_t st)
{
    if (p.n <= 0) return;
    corr_chunk_kernel<<<dim3(c.chunks.n, p.n), 32 * kSlices, 0, st>>>(d, X, c, p);
    corr_finish_kernel<<<p.n * d.n_rep, 128, 0, st>>>(d, c, p);
}

__global__ void turns_kernel(DevState d, const double *qv, int n_q, bool over_three, Turns *out)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (size_t)n_q * d.n_rep) return;
    const int r = (int)(i / n_q), k = (int)(i - (size_t)r * n_q);
    out[i] = make_turns(qv + 3 * (size_t)k, d.rep[r].h, over_three ? kInv6Pi : kInv2Pi);
}

void launch_turns(const DevState &d, const double *qv, int n_q, bool over_three, Turns *out, cudaStream_t st)
{
    turns_kernel<<<(unsigned)(((size_t)n_q * d.n_rep + 63) / 64), 64, 0, st>>>(d, qv, n_q, over_three, out);
}

// S(q): block (part, wavevector, replica) sums cos and sin of q . x over a part
// of kSqPart of the replica's records (x = q_fixed h, in [0, L); the order of
// the atoms does not matter to integer sums), then sq_sum_kernel adds the parts
// in order; out = (C^2 + S^2) / N (Eq. sq with the i = j terms included).
// Bound by the integer multiplies of the two cosines: 240 wavevectors of
// 24000 atoms took 477 us as FP64 sincos (one block per wavevector, FP64
// pipe) and take 62 us (52% of the multiply pipe).
constexpr int kSqPart = 4096;         // 16 records per thread: 32 lanes' sums of 16 stay below 2^63

__global__ void __launch_bounds__(256) sq_kernel(DevState d, int buf, const Turns *turns, int n_q, double2 *part)
{
    const int k = blockIdx.y, r = blockIdx.z;
    const RepInfo ri = d.rep[r];
    const int i0 = blockIdx.x * kSqPart, i1 = min(ri.n_sites, i0 + kSqPart);
    if (i0 >= i1) return;
    const int4 *rec = d.rec[buf] + ri.site_off;
    const Turns t = turns[(size_t)r * n_q + k];
    long long c = 0, s = 0;
    for (int i = i0 + threadIdx.x; i < i1; i += 256) {
        const int4 a = rec[i];
        const uint64_t ph = turn_phase(t, (uint32_t)a.x, (uint32_t)a.y, (uint32_t)a.z);
        c += cos_turn(ph);
        s += cos_turn(ph - (1ull << 62));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        c += __shfl_xor_sync(0xffffffffu, c, o);
        s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    __shared__ double2 red[8];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = make_double2((double)c, (double)s);
    __syncthreads();
    if (threadIdx.x == 0) {
        double2 v = red[0];
        for (int w = 1; w < 8; ++w) v = make_double2(v.x + red[w].x, v.y + red[w].y);
        part[((size_t)r * n_q + k) * gridDim.x + blockIdx.x] = v;
    }
}

__global__ void sq_sum_kernel(DevState d, const Turns *turns, int n_q, int n_part, const double2 *part, double *out,
                              int stride)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (size_t)n_q * d.n_rep) return;
    const int r = (int)(i / n_q), k = (int)(i - (size_t)r * n_q);
    const int n = d.rep[r].n_sites;
    double c = 0.0, s = 0.0;
    for (int b = 0; b * kSqPart < n; ++b) {
        const double2 v = part[i * n_part + b];
        c += v.x;
        s += v.y;
    }
    c /= kCosUnit;
    s /= kCosUnit;
    out[(size_t)r * stride + k] = turns[i].bad ? __longlong_as_double(0x7FF8000000000000ll) : (c * c + s * s) / (double)n;
}

int sq_parts(int max_sites) { return (max_sites + kSqPart - 1) / kSqPart; }

void launch_sq(const DevState &d, int buf, const Turns *turns, int n_q, int max_sites, double2 *part, double *out,
               int stride, cudaStream_t st)
{
    const int np = sq_parts(max_sites);
    sq_kernel<<<dim3(np, n_q, d.n_rep), 256, 0, st>>>(d, buf, turns, n_q, part);
    sq_sum_kernel<<<(unsigned)(((size_t)n_q * d.n_rep + 127) / 128), 128, 0, st>>>(d, turns, n_q, np, part, out, stride);
}

// Pair-distance histogram (Eq. gr): counts[b] = pairs i < j with
// floor(r / dr) = b, r from the FP64 minimum-image distance (each operation
// rounded once, in a fixed order; pair_bin64 below).
//
// What bounds it: N^2 / 2 distances.  In FP64 each takes about 12 operations
// of a pipe that does 2 per SM and cycle; a pass over the 2.9e8 pairs of 8000
// molecules took 20.4 ms.  Here the bin comes from FP32 arithmetic on the
// exact int32 differences, and FP64 decides only the pairs that FP32 cannot
// place for certain: 0.36 ms for the same pass, bound by instruction issue (36
// instructions a pair).
//
// The FP32 value of f = r / dr is within 6.5 units of 2^-24 of its own size
// (each difference rounds once when converted, three products and sums,
// sqrt.approx within 2^-23, the factor h / dr and its product), so a value
// further than 6e-7 f + 1e-6 (10 units) from a bin edge lies in the bin that
// FP64 takes.  The others (one in some thousand) compare the exact integer
// square D of the distance with the edge's, (e dr / h)^2 in FP64: both
// decisions agree unless the two are within 17 units of 2^-53 of each other,
// and inside 2^-45 the FP64 expression itself decides.
//
// Layout: blocks of 128 threads walk tile pairs of 128 x 128 records, one
// record i per thread in registers, the records j broadcast from shared
// memory.  The tile pairs of a replica are numbered by the ring distance d of
// their tiles (p = d nt + ti, partner ti + d mod nt), which meets every
// unordered pair of tiles once and needs no triangular root.  The histogram
// stays in shared memory over all tile pairs of a block; up to 1024 bins it
// is kept in four copies, by lane, because neighbouring lanes hit the same
// few bins.
constexpr int kHistTile = 128;
constexpr int kHistCopyBins = 1024;          // up to so many bins: four copies (16 KB)
constexpr int kHistBlocks = 152 * 12;        // blocks over all replicas (twelve per SM)

// the bin of one pair in FP64 (may be >= n_bins)
__device__ __noinline__ int pair_bin64(int dx, int dy, int dz, double h, double inv_h, double dr, int e)
{
    const unsigned long long D = (unsigned long long)((long long)dx * dx) + (unsigned long long)((long long)dy * dy) +
                                 (unsigned long long)((long long)dz * dz);
    const double s = (double)e * dr * inv_h;
    const double edge = s * s, diff = (double)D - edge;
    if (fabs(diff) > edge * 0x1p-45) return diff > 0.0 ? e : e - 1;
    return (int)floor(__ddiv_rn(__dsqrt_rn(r2_fixed64(dx, dy, dz, h)), dr));
}

template <int SH>
__global__ void __launch_bounds__(kHistTile) pair_hist_kernel(DevState d, int buf, double dr, int n_bins,
                                                              unsigned long long *counts)
{
    extern __shared__ unsigned int hist[];   // n_bins << SH
    __shared__ int4 tile[kHistTile];
    const int r = blockIdx.y, tid = threadIdx.x;
    const RepInfo ri = d.rep[r];
    const int N = ri.n_sites;
    const long long nt = (N + kHistTile - 1) / kHistTile, n_pairs = nt * (nt + 1) / 2;
    if (blockIdx.x >= n_pairs) return;
    const int4 *rec = d.rec[buf] + ri.site_off;
    unsigned int *mine = hist + (tid & ((1 << SH) - 1));
    for (int b = tid; b < n_bins << SH; b += kHistTile) hist[b] = 0;
    const float scale = (float)fmin(ri.h / dr, 3.0e38);
    auto flush = [&]() {
        __syncthreads();
        for (int b = tid; b < n_bins; b += kHistTile) {
            unsigned long long v = 0;
            for (int k = 0; k < 1 << SH; ++k) {
                v += hist[(b << SH) + k];
                hist[(b << SH) + k] = 0;
            }
            if (v) atomicAdd(counts + (size_t)r * n_bins + b, v);
        }
    };
    unsigned done = 0;
    for (long long p = blockIdx.x; p < n_pairs; p += gridDim.x) {
        const int dist = (int)(p / nt), ti = (int)(p - dist * nt);
        const int tj = (int)((ti + dist) % nt);
        const int i = ti * kHistTile + tid, j0 = tj * kHistTile;
        const int nj = min(kHistTile, N - j0);
        __syncthreads();
        if (tid < nj) tile[tid] = rec[j0 + tid];
        __syncthreads();
        const int4 me = rec[min(i, N - 1)];
        // one pair: place it, and count it when its bin is one of the histogram's
        auto place = [&](const int4 &o, bool on) {
            const int dx = (int)((uint32_t)o.x - (uint32_t)me.x), dy = (int)((uint32_t)o.y - (uint32_t)me.y),
                      dz = (int)((uint32_t)o.z - (uint32_t)me.z);
            const float fx = (float)dx, fy = (float)dy, fz = (float)dz;
            float root;   // (of a sum of integer squares: 0 or at least 1)
            asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(root) : "f"(fmaf(fx, fx, fmaf(fy, fy, fz * fz))));
            // bin = round(f - 1/2) by the exponent trick: 1.5 x 2^23 + g rounds
            // g to an integer, which then stands in the low bits (for g of
            // 2^22 and more, a value that exceeds every n_bins)
            const float g = fmaf(root, scale, -0.5f);
            const float t = g + 12582912.0f;
            const float off = g - (t - 12582912.0f);
            int bin = __float_as_int(t) - 0x4B400000;
            const bool near = on && bin <= n_bins;   // (the last edge may be this pair's)
            if (near && fabsf(off) > fmaf(-6e-7f, g, 0.499999f))
                bin = pair_bin64(dx, dy, dz, ri.h, ri.inv_h, dr, off > 0.f ? bin + 1 : bin);
            if (near && bin < n_bins) atomicAdd(mine + (bin << SH), 1u);
        };
        if (dist == 0) {
            for (int j = 0; j < nj; ++j) place(tile[j], j > tid && i < N);
        } else if (nj == kHistTile && (ti + 1) * kHistTile <= N) {
#pragma unroll 4
            for (int j = 0; j < kHistTile; ++j) place(tile[j], true);
        } else {
            for (int j = 0; j < nj; ++j) place(tile[j], i < N);
        }
        // a 32-bit count takes at most 2^17 tile pairs of 2^14 pairs
        if (++done == 1u << 17) {
            flush();
            done = 0;
        }
    }
    flush();
}

void launch_pair_hist(const DevState &d, int buf, int max_sites, double dr, int n_bins, unsigned long long *counts,
                      cudaStream_t st)
{
    const long long nt = (max_sites + kHistTile - 1) / kHistTile, n_pairs = nt * (nt + 1) / 2;
    const long long bx = std::min<long long>(n_pairs, std::max(1, kHistBlocks / d.n_rep));
    const dim3 grid((unsigned)bx, d.n_rep);
    if (n_bins <= kHistCopyBins)
        pair_hist_kernel<2><<<grid, kHistTile, sizeof(unsigned int) * 4 * n_bins, st>>>(d, buf, dr, n_bins, counts);
    else
        pair_hist_kernel<0><<<grid, kHistTile, sizeof(unsigned int) * n_bins, st>>>(d, buf, dr, n_bins, counts);
}

void launch_gather(const DevState &d, int buf, long long *X, int *types, cudaStream_t st)
{
    gather_kernel<<<(d.n_sites + 255) / 256, 256, 0, st>>>(d, buf, X, types);
}

void launch_set_t0(const DevState &d, const long long *X, const int *types, const ObsState &o, cudaStream_t st)
{
    const int nm = d.n_sites / 3;
    set_t0_kernel<<<(nm + 127) / 128, 128, 0, st>>>(d, X, types, o);
}

void launch_observables(const DevState &d, const long long *X, const ObsState &o, const MolChunks &mc, const Turns *ta,
                        int nqa, const Turns *tc, int nqc, double *fs_site, double *fscm_mol, double *c2_mol,
                        double *part, double *out, cudaStream_t st)
{
    observables_kernel<<<mc.n, 32 * kSlices, 0, st>>>(d, X, o, mc, ta, nqa, tc, nqc, fs_site, fscm_mol, c2_mol, part);
    observables_mean_kernel<<<d.n_rep, 128, 0, st>>>(d, mc, part, out);
}

}  // namespace flipmc
