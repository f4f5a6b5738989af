// cd_pack_core.cuh -- the caller's velocities into the sweep state (Eq. 1),
// shared by the kernels that do it.
#pragma once

#include "cd_sweep_core.cuh"

// ---------------------------------------------------------------------------
// Packs the caller's velocities into the sweep state; with free_flight the
// explicit external forces of Eq. 1 are applied first (F = m g + f_ext).
// ---------------------------------------------------------------------------
// block0: this block packs the force-controlled walls.
template <int DIM, typename T>
__device__ __forceinline__ void pack_velocities(const CdGeom& g, const CdWork& w, const double* __restrict__ vel,
                                                const double* __restrict__ omega, const double* __restrict__ inv_m,
                                                const double* __restrict__ f_ext, int free_flight, int tid, int stride,
                                                bool block0)
{
    typedef typename Vec<T>::V4 T4;
    T4* V = (T4*)w.V;
    // force-controlled walls: velocity records n + k, pushed along the inward normal (Eq. 1)
    if (g.dyn_walls && block0 && threadIdx.x < 6 && ((g.dyn_walls >> threadIdx.x) & 1)) {
        const int k = threadIdx.x, ax = k >> 1;
        double u[3] = {w.pk[0].wall_vel[3 * k], w.pk[0].wall_vel[3 * k + 1], w.pk[0].wall_vel[3 * k + 2]};
        if (free_flight) {
            double a = __dmul_rn(g.wall_push[k], g.wall_im[k]);
            if (k & 1) a = -a;
            u[ax] = __dadd_rn(u[ax], __dmul_rn(a, g.dt));
        }
        T4 s;
        s.x = (T)u[0]; s.y = (T)u[1]; s.z = (T)((DIM == 3) ? u[2] : 0.0); s.w = (T)0;
        if (DIM == 2) {
            V[g.n + k] = s;
        } else {
            T4 o;
            o.x = (T)0; o.y = (T)0; o.z = (T)0; o.w = (T)0;
            V[2 * (g.n + k)] = s;
            V[2 * (g.n + k) + 1] = o;
        }
    }
    for (int i = tid; i < g.n; i += stride) {
        double v[3] = {0.0, 0.0, 0.0};
        double im = inv_m[i];
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            double vk = vel[i * DIM + k];
            if (free_flight) {
                double gk = (g.npk > 1) ? w.pk[w.pack_of[i]].gravity[k] : g.gravity[k];
                double a = (im == 0.0) ? 0.0 : gk;
                if (f_ext) a = __dadd_rn(a, __dmul_rn(f_ext[i * DIM + k], im));
                vk = __dadd_rn(vk, __dmul_rn(a, g.dt));
            }
            v[k] = vk;
        }
        if (DIM == 2) {
            T4 s;
            s.x = (T)v[0]; s.y = (T)v[1]; s.z = (T)omega[i]; s.w = (T)0;
            V[i] = s;
        } else {
            T4 s, o;
            s.x = (T)v[0]; s.y = (T)v[1]; s.z = (T)v[2]; s.w = (T)0;
            o.x = (T)omega[3 * i]; o.y = (T)omega[3 * i + 1]; o.z = (T)omega[3 * i + 2]; o.w = (T)0;
            V[2 * i] = s;
            V[2 * i + 1] = o;
        }
    }
}

// Particle i's velocities (v, o: its record) to the caller's arrays; with
// integrate its position (and 2D orientation) follows Eq. 2.
template <int DIM, typename T>
__device__ __forceinline__ void unpack_particle(const CdGeom& g, const CdState& io, int i, const typename Vec<T>::V4& s,
                                                const typename Vec<T>::V4& o)
{
    const double v[3] = {(double)s.x, (double)s.y, DIM == 3 ? (double)s.z : 0.0};
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        io.vel[i * DIM + k] = v[k];
        if (io.integrate) {
            double xn = __dadd_rn(io.pos[i * DIM + k], __dmul_rn(v[k], g.dt));
            if (g.periodic[k]) {
                if (xn >= g.hi[k]) xn = __dsub_rn(xn, g.L[k]);
                else if (xn < g.lo[k]) xn = __dadd_rn(xn, g.L[k]);
            }
            io.pos[i * DIM + k] = xn;
        }
    }
    if (DIM == 2) {
        const double om = (double)s.z;
        io.omega[i] = om;
        if (io.integrate && io.theta) io.theta[i] = __dadd_rn(io.theta[i], __dmul_rn(om, g.dt));
    } else {
        io.omega[3 * i] = (double)o.x; io.omega[3 * i + 1] = (double)o.y; io.omega[3 * i + 2] = (double)o.z;
    }
}

// Force-controlled walls: their velocity after the solve becomes the wall velocity.
template <int DIM, typename T>
__device__ __forceinline__ void unpack_walls(const CdGeom& g, const CdWork& w)
{
    typedef typename Vec<T>::V4 T4;
    const T4* V = (const T4*)w.V;
    for (int k = 0; k < 2 * DIM; ++k) {
        if (!((g.dyn_walls >> k) & 1)) continue;
        const T4 s = (DIM == 2) ? V[g.n + k] : V[2 * (g.n + k)];
        const double u[3] = {(double)s.x, (double)s.y, (double)s.z};
        w.pk[0].wall_vel[3 * k + (k >> 1)] = u[k >> 1];
    }
}

// The walls of packing b move (Eq. 2).
template <int DIM>
__device__ __forceinline__ void move_walls(const CdGeom& g, const CdWork& w, int b)
{
    const CdPack& pb = w.pk[b];
    for (int k = 0; k < 2 * DIM; ++k)
        if ((pb.wall_mask >> k) & 1)
            w.pk_wall_pos[6 * b + k] =
                __dadd_rn(w.pk_wall_pos[6 * b + k], __dmul_rn(pb.wall_vel[3 * k + (k >> 1)], g.dt));
}
