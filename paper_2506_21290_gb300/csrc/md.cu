// Molecular dynamics of the flexible three-site molecules (Sec. II.D: NVT,
// time step 0.001, Nose-Hoover thermostat with relaxation time 1), FP64.
//
// One step, a symmetric (time-reversible) splitting of velocity Verlet and
// the thermostat, m = 1, g = 3N degrees of freedom, Q = g T tau^2:
//   xi += dt/2 (2K - gT) / Q;  eta += dt/2 xi;  v *= exp(-xi dt/2);  v += dt/2 F
//   q  += rint(v dt / h)                     (fixed point, periodic images counted)
//   cell list; F = forces (Eq. 1 and 2, every pair inside its range)
//   v += dt/2 F;  v *= exp(-xi dt/2);  xi += dt/2 (2K - gT) / Q;  eta += dt/2 xi
// K is the kinetic energy sum v^2 / 2 over the replica, in a fixed order.  The
// conserved quantity is K + U + Q xi^2 / 2 + g T eta.
//
// A step is five kernels, seven above 8192 cells: the move (kick, drift and the
// count of the cell list), its scan (one kernel or three), scatter and order, and
// the forces, whose blocks end the step for their atoms.  The kinetic energy at
// the start of a step is the one at the end of the step before, so the block that
// is the last of its replica to finish takes both thermostat half steps.  (As
// thirteen kernels, with K summed twice, the parts beside the forces took 45 us a
// step at 1000 molecules and 70 at 64000.)
#include "cell_list.h"
#include "cell_list_dev.cuh"
#include "flipmc_device.cuh"
#include "md.h"
#include "pair_walk.cuh"

namespace flipmc {

// First kick and drift of one record per thread, and its count in the new
// position's cell.
__global__ void __launch_bounds__(256) md_move_kernel(DevState d, int buf, MdDev m)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= d.n_sites) return;
    const int r = d.rep_of_site[g];
    const RepInfo ri = d.rep[r];
    int4 rc = d.rec[buf][g];
    const size_t site = ri.site_off + rec_site(rc.w);
    const double sc = m.scale[r];
    const double s = m.dt * ri.inv_h;   // fixed-point units per unit velocity and step
    uint32_t q3[3] = {(uint32_t)rc.x, (uint32_t)rc.y, (uint32_t)rc.z};
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const double v = __dadd_rn(__dmul_rn(m.v[3 * site + ax], sc), __dmul_rn(m.hdt, m.F[3 * site + ax]));
        m.v[3 * site + ax] = v;
        const long long moved = (long long)q3[ax] + (long long)rint(__dmul_rn(v, s));
        if (moved < 0) d.img[3 * site + ax] -= 1;
        else if (moved >= 4294967296ll) d.img[3 * site + ax] += 1;
        q3[ax] = (uint32_t)moved;
    }
    rc.x = (int)q3[0];
    rc.y = (int)q3[1];
    rc.z = (int)q3[2];
    d.rec[buf][g] = rc;
    cl_count_item(d, buf, g, d.ctr[r].sweep, d.cell_count);
}

// The pair factor (-r dphi/dr) / r^2 in FP32: r^2 from the exact int32
// differences (one rounding per axis), the derivative of Eq. 1 and Eq. 2.
__device__ __forceinline__ float virial_over_r2_f32(const ModelDev &md, float r2, int ab, bool bonded)
{
    const float inv = 1.0f / r2;
    float w = 0.f;
    if (r2 < md.rc2f[ab]) {
        const float t = md.s2f[ab] * inv;
        const float s6 = t * t * t;
        w = 6.0f * md.e4f * s6 * (2.0f * s6 - 1.0f);
    }
    if (bonded) {
        const float x = r2 * md.invR2f[ab];
        w += 2.0f * md.nkef * x / (1.0f - x);
    }
    return w * inv;
}

// Both thermostat half steps that follow from K (one thread): the end of this
// step (unless it is the setup) and the start of the next.
__device__ void md_thermostat(const DevState &d, const MdDev &m, int r, double v2, bool end_step)
{
    const double g = 3.0 * (double)d.rep[r].n_sites;
    const double a = __dmul_rn(m.hdt, __ddiv_rn(__dsub_rn(v2, g * m.T[r]), m.Q[r]));   // 2 K = v2
    double xi = m.xi[r], eta = m.eta[r];
    if (end_step) {
        xi = __dadd_rn(m.xi_mid[r], a);
        eta = __dadd_rn(m.eta_mid[r], __dmul_rn(m.hdt, xi));
        m.xi[r] = xi;
        m.eta[r] = eta;
    }
    xi = __dadd_rn(xi, a);
    m.xi_mid[r] = xi;
    m.eta_mid[r] = __dadd_rn(eta, __dmul_rn(m.hdt, xi));
    m.scale[r] = exp(-xi * m.hdt);
}

// The end of a step for component c of a site: second kick; returns v^2.
__device__ __forceinline__ double md_second_kick(const MdDev &m, size_t o, double F, double scale)
{
    const double v = __dmul_rn(__dadd_rn(m.v[o], __dmul_rn(m.hdt, F)), scale);
    m.v[o] = v;
    return __dmul_rn(v, v);
}

// Fixed-order sum over nb partial sums by T threads (red: T doubles in shared
// memory): four chains per thread, then a tree.  All threads call; thread 0 gets it.
template <int T>
__device__ __forceinline__ double sum_parts(const double *part, int nb, double *red)
{
    const int tid = threadIdx.x;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (int k = tid; k < nb; k += 4 * T)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (k + j * T < nb) s[j] = __dadd_rn(s[j], __ldcg(part + k + j * T));
    red[tid] = __dadd_rn(__dadd_rn(s[0], s[1]), __dadd_rn(s[2], s[3]));
    __syncthreads();
    for (int o = T / 2; o > 0; o >>= 1) {
        if (tid < o) red[tid] = __dadd_rn(red[tid], red[tid + o]);
        __syncthreads();
    }
    return red[0];
}

// The last of a replica's nb blocks to get here, with all their parts visible,
// gets true; it leaves the counter at zero.  All threads call; the block's own
// part was written by thread 0.  The counter is the MD run's own, whose steps
// follow one another.
__device__ __forceinline__ bool last_block(unsigned *arrived, int nb)
{
    __shared__ int last;
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(arrived, 1u) == (unsigned)nb - 1u;
        if (last) {
            *arrived = 0;
            __threadfence();
        }
    }
    __syncthreads();
    return last != 0;
}

// The end of a step for a block: its sum of v^2 (every thread's share), and by
// the replica's last block the thermostat; clears the cell counts for the next step.
template <int T>
__device__ void md_end_step(const DevState &d, const MdDev &m, int r, int b0, int nb, double v2, double *red)
{
    for (int c = blockIdx.x * T + threadIdx.x; c < d.n_cells; c += gridDim.x * T) d.cell_count[c] = 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v2 = __dadd_rn(v2, __shfl_xor_sync(0xffffffffu, v2, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v2;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < T / 32; ++k) v2 = __dadd_rn(v2, red[k]);
        m.part[blockIdx.x] = v2;
    }
    if (!last_block(m.arrived + r, nb)) return;
    v2 = sum_parts<T>(m.part + b0, nb, red);
    if (threadIdx.x == 0) md_thermostat(d, m, r, v2, true);
}

// FP64 forces: F_i = sum over partners j of (-r dphi/dr) / r^2 (x_i - x_j),
// partners in the neighbour cells in cell order, then record order.  One warp
// per cell (pair_walk.cuh).  The evaluated pairs' contributions go to a list in
// shared memory in that order; lane 3 i + axis then adds up atom i's share of the
// list, one after the other, so the sum is the same on every run.
// With one thread per atom, 10 of 32 lanes were active in an evaluation, and 94
// warps had 3000 atoms: 294 us at 1000 molecules, now 23 (latency: at 8 warps an SM
// or fewer nothing fills the FP64 chains).  Against extended precision the forces
// are 1.55e-15 of their norm off (1.85e-15 with divisions and h applied per axis).
constexpr int kMdList = 128;       // contributions waiting per warp

struct ForceWalk {
    const RepInfo &ri;
    const ModelDev &md;
    const MdDev &m;
    const int4 *ring;
    double (*list)[kMdList];       // the three components
    int *first;                    // [33] position of each own atom's first pair
    const int lane;
    const Quantum2 hh;
    const double scale;
    const bool end_step;
    int n_own = 0, cur = 0, flushed = 0, own_w = 0;
    double acc[3] = {0, 0, 0};     // component lane + 32 j of the own atoms' forces
    double v2 = 0.0;

    __device__ void own(int, int ni, const int4 &rec)
    {
        n_own = ni;
        own_w = rec.w;
        acc[0] = acc[1] = acc[2] = 0;
    }
    __device__ void atom(int i, int at)
    {
        cur = i;
        if (lane == 0) first[i] = at;
    }
    // add the list's pairs up to position `to` to their atoms
    __device__ void flush(int to)
    {
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int t = lane + 32 * j, i = t / 3, c = t - 3 * i;
            if (32 * j <= 3 * cur + 2 && i <= cur) {
                const int lo = max(first[i], flushed) - flushed, hi = (i == cur ? to : min(first[i + 1], to)) - flushed;
                double a = acc[j];
                for (int e = lo; e < hi; ++e) a = __dsub_rn(a, list[c][e]);
                acc[j] = a;
            }
        }
        flushed = to;
        __syncwarp();
    }
    __device__ void eval(int at, int n)
    {
        if (at + 32 - flushed > kMdList) flush(at);
        if (lane < n) {
            const int4 e = ring[(at + lane) & (kWalkRing - 1)];
            const int ab = walk_types(e.w), o = at - flushed + lane;
            const double r2 = walk_r2(e, hh);
            const double inv = walk_rcp(r2);
            const double t = md.s2[ab] * inv;
            const double s6 = t * t * t;
            double w = r2 < md.rc2[ab] ? 6.0 * md.e4 * (s6 * fma(2.0, s6, -1.0)) * inv : 0.0;
            // FENE, -2 K eps x / (1 - x) with x = r^2 / R^2, over r^2
            if (walk_bonded(e.w)) w = fma(2.0 * md.nke * md.invR2[ab], walk_rcp(1.0 - r2 * md.invR2[ab]), w);
            w *= ri.h;
            list[0][o] = w * (double)e.x;
            list[1][o] = w * (double)e.y;
            list[2][o] = w * (double)e.z;
        }
    }
    __device__ void part(int &head, int tail)
    {
        if (tail > head) eval(head, tail - head);
        head = tail;
        flush(tail);
    }
    // the forces of the own atoms and, at the end of a step, their second kick
    __device__ void done()
    {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int t = lane + 32 * j, i = t / 3, c = t - 3 * i;
            const int w = __shfl_sync(0xffffffffu, own_w, i & 31);
            if (i < n_own) {
                const size_t o = 3 * (size_t)(ri.site_off + rec_site(w)) + c;
                m.F[o] = acc[j];
                if (end_step) v2 = __dadd_rn(v2, md_second_kick(m, o, acc[j], scale));
            }
        }
    }
};

// end_step: 1 ends a step; 0 only computes the forces (setup: the velocities are
// the user's, and K is theirs).
__global__ void __launch_bounds__(32 * kMdWarps, 4) md_force64_kernel(DevState d, int buf, MdDev m, int end_step)
{
    __shared__ WalkSmem walk[kMdWarps];
    __shared__ double list[kMdWarps][3][kMdList], red[32 * kMdWarps];
    __shared__ int first[kMdWarps][33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int2 u = m.units.unit[blockIdx.x];
    const RepInfo ri = d.rep[u.x];
    ForceWalk p{ri, *d.model, m, walk[w].ring, list[w], first[w], lane, quantum2(ri.h), m.scale[u.x], end_step != 0};
    int head = 0, tail = 0;
    const int n_cells = ri.nc * ri.nc * ri.nc;
    const MdWarps mw = md_warps(ri.n_sites, n_cells);
    const int id = u.y + w;        // warp of the replica
    const int cell = id / mw.slices, c0 = ri.cell_off + cell * mw.cells;
    unsigned todo = cell < n_cells ? 1u : 0u;   // cells c0 + bit
    if (mw.cells > 1) {
        const int c = c0 + lane;
        const bool full = lane < mw.cells && c < ri.cell_off + n_cells && d.cell_start[c + 1] > d.cell_start[c];
        todo = __ballot_sync(0xffffffffu, full);
    }
    for (; todo != 0; todo &= todo - 1)
        walk_cell<false, true>(d, ri, *d.model, d.rec[buf], c0 + __ffs(todo) - 1, lane, walk[w], head, tail, p,
                               id - cell * mw.slices, mw.slices);
    const int b0 = m.units.rep0[u.x];
    if (end_step) md_end_step<32 * kMdWarps>(d, m, u.x, b0, m.units.rep0[u.x + 1] - b0, p.v2, red);
}

// FP32 forces (pair terms and their sums in FP32, from the exact differences),
// one thread per atom, in the order of the neighbour cells (x fastest) and
// records.  The three cells of a row along x lie end to end in the records (two
// runs where the row wraps around the box), so the 27 cells are 9 to 18 runs,
// whose extents are fetched first.  A thread notes its hits in a list in shared
// memory (no branch: the place after the last hit takes what is none) and
// evaluates the list when it is through: evaluated where they are found, the hits
// of a warp's atoms fall into nearly every iteration, with a few lanes active in
// each.  192000 atoms 86 us (99); the warp-per-cell walk with a list of
// contributions took 180 (16 warps per SM).
constexpr int kHitList = 32;

struct HitSmem {
    int list[kHitList + 1][32];    // records of the hits, a column per lane
    int run[18][32], len[18][32];  // runs of candidate records: the first, and how many
};

// the runs of candidates around `me` into this lane's column; returns how many
__device__ __forceinline__ int md_runs(const DevState &d, const RepInfo &ri, const uint32_t *shift, const int4 &me, HitSmem &sm)
{
    const int lane = threadIdx.x & 31, nc = ri.nc;
    const int cx = (int)cell_axis((uint32_t)me.x, shift[0], nc), cy = (int)cell_axis((uint32_t)me.y, shift[1], nc),
              cz = (int)cell_axis((uint32_t)me.z, shift[2], nc);
    const bool small = nc == 2;
    // the cells [x0, x1) of a row's first run and [0, x2) of its second
    int x0 = cx - 1, x1 = cx + 2, x2 = 0;
    if (small) {
        x0 = cx;
        x1 = 2;
        x2 = cx;
    } else if (cx == 0) {
        x0 = nc - 1;
        x1 = nc;
        x2 = 2;
    } else if (cx == nc - 1) {
        x1 = nc;
        x2 = 1;
    }
    int n_run = 0, a[9], b[9], la[9], lb[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        la[k] = lb[k] = 0;
        if (k < 4 || !small) {
            int y = small ? cy + (k & 1) : cy + k % 3 - 1, z = small ? cz + (k >> 1) : cz + k / 3 - 1;
            y += y < 0 ? nc : (y >= nc ? -nc : 0);
            z += z < 0 ? nc : (z >= nc ? -nc : 0);
            const int *start = d.cell_start + ri.cell_off + (z * nc + y) * nc;
            a[k] = start[x0];
            la[k] = start[x1] - a[k];
            if (x2 > 0) {
                b[k] = start[0];
                lb[k] = start[x2] - b[k];
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        if (la[k] > 0) {
            sm.run[n_run][lane] = a[k];
            sm.len[n_run++][lane] = la[k];
        }
        if (lb[k] > 0) {
            sm.run[n_run][lane] = b[k];
            sm.len[n_run++][lane] = lb[k];
        }
    }
    return n_run;
}

__global__ void __launch_bounds__(32) md_force32_kernel(DevState d, int buf, MdDev m, int end_step)
{
    __shared__ HitSmem sm;
    __shared__ double red[32];
    const int lane = threadIdx.x;
    const int2 u = m.units.unit[blockIdx.x];
    const RepInfo ri = d.rep[u.x];
    const ModelDev &md = *d.model;
    double v2 = 0.0;
    if (u.y + lane < ri.site_off + ri.n_sites) {
        const int4 *rec = d.rec[buf];
        const int4 me = rec[u.y + lane];
        const int n_run = md_runs(d, ri, d.ctr[u.x].shift, me, sm);
        const int t3 = 3 * rec_type(me.w);
        // the own type's largest cutoff, fixed-point units squared, with a margin
        // of 2e-5 on r^2: what is left out contributes exactly 0
        const float cut = fmaxf(md.rc2f[t3], fmaxf(md.rc2f[t3 + 1], md.rc2f[t3 + 2])) * 1.00002f / ri.hf / ri.hf;
        float gx = 0.f, gy = 0.f, gz = 0.f;
        int k = 0, t = 0, first = sm.run[0][lane], len = sm.len[0][lane];   // (its own cell's run is never empty)
        do {
            int n = 0;
            while (k < n_run && n <= kHitList - 4) {
                int4 o[4];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (t + q < len) o[q] = rec[first + t + q];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float fx = (float)(int)((uint32_t)o[q].x - (uint32_t)me.x),
                                fy = (float)(int)((uint32_t)o[q].y - (uint32_t)me.y),
                                fz = (float)(int)((uint32_t)o[q].z - (uint32_t)me.z);
                    const uint32_t x = (uint32_t)(o[q].w ^ me.w);   // below 16: the same molecule, below 4: the atom
                    sm.list[n][lane] = first + t + q;
                    n += ((fmaf(fx, fx, fmaf(fy, fy, fz * fz)) <= cut) | (x < 16u)) & (x >= 4u) & (t + q < len);
                }
                t += 4;
                if (t >= len && ++k < n_run) {
                    t = 0;
                    first = sm.run[k][lane];
                    len = sm.len[k][lane];
                }
            }
#pragma unroll 2
            for (int e = 0; e < n; ++e) {
                const int4 o = rec[sm.list[e][lane]];
                const float ex = (float)(int)((uint32_t)o.x - (uint32_t)me.x) * ri.hf,
                            ey = (float)(int)((uint32_t)o.y - (uint32_t)me.y) * ri.hf,
                            ez = (float)(int)((uint32_t)o.z - (uint32_t)me.z) * ri.hf;
                const float w = virial_over_r2_f32(md, fmaf(ex, ex, fmaf(ey, ey, ez * ez)), t3 + rec_type(o.w),
                                                   (uint32_t)(o.w ^ me.w) < 16u);
                gx = fmaf(-w, ex, gx);
                gy = fmaf(-w, ey, gy);
                gz = fmaf(-w, ez, gz);
            }
        } while (k < n_run);
        const double F[3] = {(double)gx, (double)gy, (double)gz}, scale = m.scale[u.x];
        const size_t o = 3 * (size_t)(ri.site_off + rec_site(me.w));
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            m.F[o + c] = F[c];
            if (end_step) v2 = __dadd_rn(v2, md_second_kick(m, o + c, F[c], scale));
        }
    }
    const int b0 = m.units.rep0[u.x];
    if (end_step) md_end_step<32>(d, m, u.x, b0, m.units.rep0[u.x + 1] - b0, v2, red);
}

// Setup: K of the initial velocities (one block per replica, fixed order) and
// the first thermostat half step.
__global__ void __launch_bounds__(512) md_start_kernel(DevState d, MdDev m)
{
    const int r = blockIdx.x, tid = threadIdx.x;
    const RepInfo ri = d.rep[r];
    const double *v = m.v + 3 * (size_t)ri.site_off;
    double s = 0.0;
    for (size_t k = tid; k < 3 * (size_t)ri.n_sites; k += 512) s = __dadd_rn(s, __dmul_rn(v[k], v[k]));
    __shared__ double red[512];
    red[tid] = s;
    __syncthreads();
    for (int o = 256; o > 0; o >>= 1) {
        if (tid < o) red[tid] = __dadd_rn(red[tid], red[tid + o]);
        __syncthreads();
    }
    if (tid == 0) md_thermostat(d, m, r, red[0], false);
}

static void launch_forces(const DevState &d, int buf, const MdDev &m, int end_step, cudaStream_t st)
{
    if (m.fp32_forces) md_force32_kernel<<<m.units.n, 32, 0, st>>>(d, buf, m, end_step);
    else md_force64_kernel<<<m.units.n, 32 * kMdWarps, 0, st>>>(d, buf, m, end_step);
}

void launch_md_setup(const DevState &d, int buf, const MdDev &m, cudaStream_t st)
{
    md_start_kernel<<<d.n_rep, 512, 0, st>>>(d, m);
    launch_md_forces(d, buf, m, st);
}

void launch_md_forces(const DevState &d, int buf, const MdDev &m, cudaStream_t st)
{
    launch_forces(d, buf, m, 0, st);
}

void launch_md_step(const DevState &d, int buf, const MdDev &m, cudaStream_t st)
{
    md_move_kernel<<<(d.n_sites + 255) / 256, 256, 0, st>>>(d, buf, m);
    launch_cell_sort(d, buf, buf ^ 1, st);
    launch_forces(d, buf ^ 1, m, 1, st);
}

}  // namespace flipmc
