// Langevin dynamics on the device (BAOAB splitting, Leimkuhler and Matthews): every
// configuration of a batch advances its own trajectory; the potential is the PANNA
// energy/force path of the rest of the library (Sec. II), evaluated once per step.  The
// paper times Langevin MD on a small carbon cell (Sec. III.B); it does not name the
// integrator.
//
// Units: positions A, velocities A/fs, time fs, masses amu, energies eV, temperature K.
// The noise is Philox4x32-10 (Salmon, Moraes, Dror and Shaw, SC'11) with counter
// (atom, step) and key seed, turned into normals by Box-Muller, so a trajectory does not
// depend on the launch shape.
#include "common.cuh"

namespace panna {

// Philox4x32-10: ten rounds of two 32 x 32 -> 64-bit products on words 0 and 2 of the
// counter, the high halves mixed with words 1, 3 and the key, the key advanced by two Weyl
// constants between rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k)
{
    const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u, W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) { k.x += W0; k.y += W1; }
        const uint32_t hi0 = __umulhi(M0, c.x), lo0 = M0 * c.x;
        const uint32_t hi1 = __umulhi(M1, c.z), lo1 = M1 * c.z;
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    }
    return c;
}

// component d of the three standard normals of atom a at step t: Box-Muller on u = (x + 1/2) 2^-32,
// components 0 and 1 from the first two words, 2 from the others
__device__ __forceinline__ double gauss_component(uint64_t seed, int64_t a, int64_t t, int d)
{
    const uint4 x = philox4x32_10(make_uint4((uint32_t)a, (uint32_t)((uint64_t)a >> 32), (uint32_t)t,
                                             (uint32_t)((uint64_t)t >> 32)),
                                  make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
    const double s32 = 1.0 / 4294967296.0;
    const double u = ((double)(d < 2 ? x.x : x.z) + 0.5) * s32, w = ((double)(d < 2 ? x.y : x.w) + 0.5) * s32;
    double sn, cs;
    sincospi(2.0 * w, &sn, &cs);
    return sqrt(-2.0 * log(u)) * (d == 1 ? sn : cs);
}

// (B of the step before when pending) B A O A: v += dt/2 a F; x += dt/2 v; v = c1 v + c2 sigma g;
// x += dt/2 v.  Four lanes per atom, one per component: the normals' FP64 logarithm, root and sine are
// the kernel's time (one lane per atom took all three in turn: 10 -> 8 us).  With a reference (positions
// of the last neighbour build), an atom that has moved more than sqrt(lim2) since then raises *stale,
// and the positions folded with the lattice offsets of that build (wrap) go to pos_hi / pos_lo for the
// list's refresh, so the image shifts stored with the candidates stay valid while atoms move.
__global__ void k_md_baoa(int64_t N, const int32_t* __restrict__ species, MdSpecies ms, double* __restrict__ pos,
                          double* __restrict__ vel, const float* __restrict__ F, double dt, double c1, double c2,
                          int thermostat, uint64_t seed, int64_t step, int pending_b,
                          const double* __restrict__ pos_ref, double lim2, int32_t* __restrict__ stale,
                          const int32_t* __restrict__ atom_cfg, const CfgGeom* __restrict__ geom,
                          const int32_t* __restrict__ wrap, float4* __restrict__ pos_hi, float4* __restrict__ pos_lo)
{
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, i = idx >> 2;
    const int lane = threadIdx.x & 31, d = lane & 3, q = lane & ~3;
    const bool on = i < N;
    double x = 0.0, e2 = 0.0;
    if (on && d < 3) {
        const int sp = species[i];
        const double a = ms.acc[sp], f = 0.5 * dt * (double)F[3 * i + d] * a;
        double v = vel[3 * i + d];
        if (pending_b) v += f;
        v += f;
        x = pos[3 * i + d] + 0.5 * dt * v;
        if (thermostat) v = c1 * v + c2 * ms.sigma[sp] * gauss_component(seed, i, step, d);
        x += 0.5 * dt * v;
        vel[3 * i + d] = v;
        pos[3 * i + d] = x;
        const double e = x - pos_ref[3 * i + d];
        e2 = e * e;
    }
    float h = 0.f, l = 0.f;
    if (on && d < 3) {
        const CfgGeom& g = geom[atom_cfg[i]];
        const double xw = x + wrap[3 * i] * g.cell[d] + wrap[3 * i + 1] * g.cell[3 + d] + wrap[3 * i + 2] * g.cell[6 + d];
        h = (float)xw;
        l = (float)(xw - h);
    }
    const double s0 = __shfl_sync(0xffffffffu, e2, q), s1 = __shfl_sync(0xffffffffu, e2, q + 1),
                 s2 = __shfl_sync(0xffffffffu, e2, q + 2);
    const float h1 = __shfl_sync(0xffffffffu, h, q + 1), h2 = __shfl_sync(0xffffffffu, h, q + 2);
    const float l1 = __shfl_sync(0xffffffffu, l, q + 1), l2 = __shfl_sync(0xffffffffu, l, q + 2);
    if (on && d == 0) {
        if ((s0 + s1) + s2 > lim2) *stale = 1;
        pos_hi[i] = make_float4(h, h1, h2, pos_hi[i].w);
        pos_lo[i] = make_float4(l, l1, l2, 0.f);
    }
}

// B: v += dt/2 a F
__global__ void k_md_b(int64_t N, const int32_t* __restrict__ species, MdSpecies ms, double* __restrict__ vel,
                       const float* __restrict__ F, double dt)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double a = ms.acc[species[i]];
#pragma unroll
    for (int d = 0; d < 3; ++d) vel[3 * i + d] += 0.5 * dt * (double)F[3 * i + d] * a;
}

cudaError_t launch_md_baoa(const Work& w, const MdSpecies& ms, double* pos, double* vel, const float* F, double dt,
                           double c1, double c2, int thermostat, uint64_t seed, int64_t step, bool pending_b,
                           const double* pos_ref, double lim2, cudaStream_t s)
{
    if (w.N == 0) return cudaSuccess;
    k_md_baoa<<<(unsigned)((4 * w.N + 255) / 256), 256, 0, s>>>(w.N, w.sys->species, ms, pos, vel, F, dt, c1, c2,
                                                                thermostat, seed, step, pending_b ? 1 : 0, pos_ref,
                                                                lim2, &w.status->stale, w.atom_cfg, w.geom, w.wrap,
                                                                w.pos_hi, w.pos_lo);
    return cudaGetLastError();
}

cudaError_t launch_md_b(int64_t N, const int32_t* species, const MdSpecies& ms, double* vel, const float* F,
                        double dt, cudaStream_t s)
{
    if (N == 0) return cudaSuccess;
    k_md_b<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(N, species, ms, vel, F, dt);
    return cudaGetLastError();
}

}  // namespace panna
