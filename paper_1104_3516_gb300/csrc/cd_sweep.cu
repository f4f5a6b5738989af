// cd_sweep.cu -- the iterative contact-impulse solve (paper Sec. 2.1, Fig. 2)
// and the Euler update (Eqs. 1-2).
//
// Long solves of plain systems, the domain-wise update and most batches run as a
// dataflow instead (cd_flow.cu).
//
// k_sweep is one cooperative persistent launch per solve: it applies the
// starting impulses, then repeats sweeps over the colour classes (one grid
// barrier per colour) until the convergence test of Sec. 2.1 passes or the
// sweep cap is hit.  All blocks compute the residual from the same per-block
// partial sums in the same order, so they agree on when to stop without any
// host round trip.
//
// Single-contact update (Fig. 2), in impulses P = R dt.  With u the current
// relative velocity of the contact points (this contact's own impulse
// included) and M = diag(m_n, m_t) the pair mass matrix (Eq. 5), removing the
// own impulse gives v_g0 = u - M^-1 P_old, so the sticking impulse of Eq. 5,
// P = -M (g/dt n + v_g0), reads
//     P_n* = P_n,old - m_n (g/dt + u_n),   P_t* = P_t,old - m_t u_t.
// Eq. 3 (gap stays open) is P_n* < 0 -> P = 0; the Coulomb test (Eq. 8) and
// the sliding solution (Eqs. 9-11: tangential impulse of magnitude mu P_n
// against the sliding velocity, which for discs and spheres is parallel to
// P_t*) give P_t = P_t* scaled onto |P_t| <= mu P_n.
#include <type_traits>

#include "cd_pack_core.cuh"

// Variants of the persistent colour-barrier sweep: plain Gauss-Seidel, the
// mixed update of Sec. 2.3, the domain-wise update of Sec. 3.1.
enum { CD_SWEEP_PLAIN = 0, CD_SWEEP_MIXED = 1, CD_SWEEP_DOMAINS = 2, CD_SWEEP_MERGE = 3 };

// Merged last phase of a step (params.merge_last_colour): phase `klast` runs
// the M last colours in place of M phases.  This block's positions of colour
// K-M+m are mg_list[lst[2m] .. lst[2m + 1]) (lst in shared memory).  The
// block's items are numbered through the M lists in turn;
// item q goes to thread q % blockDim, so a thread's first item (prefetched
// before the grid barrier) may belong to any of the lists, and the later
// sub-steps wait after their block barrier only for their velocities.
struct MgInfo {
    int on;
    int klast;
    int M;
    const int* lst;
    long long draw;   // mixed update: the iteration step whose parallel subset applies (-1: fixed subset)
};

// ---------------------------------------------------------------------------
// Static per-particle record (inv_m, r, r / I, 0) in the sweep's real type.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_static(CdGeom g, int n, int rotations, const double* __restrict__ radius,
                         const double* __restrict__ inv_m, const double* __restrict__ inv_I,
                         typename Vec<T>::V4* __restrict__ S)
{
    // records n .. n + 5: force-controlled walls (inverse mass, no radius, no rotation)
    if (blockIdx.x == 0 && threadIdx.x < 6) {
        typename Vec<T>::V4 s;
        s.x = (T)(((g.dyn_walls >> threadIdx.x) & 1) ? g.wall_im[threadIdx.x] : 0.0);
        s.y = (T)0; s.z = (T)0; s.w = (T)0;
        S[n + threadIdx.x] = s;
    }
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        typename Vec<T>::V4 s;
        double r = radius[i];
        s.x = (T)inv_m[i];
        s.y = (T)r;
        s.z = rotations ? (T)(r * inv_I[i]) : (T)0;
        s.w = (T)0;
        S[i] = s;
    }
}

template <int DIM, typename T>
__global__ void k_pack(CdGeom g, CdWork w, const double* __restrict__ vel, const double* __restrict__ omega,
                       const double* __restrict__ inv_m, const double* __restrict__ f_ext, int free_flight)
{
    if (w.ctrl->skip) return;
    pack_velocities<DIM, T>(g, w, vel, omega, inv_m, f_ext, free_flight, blockIdx.x * blockDim.x + threadIdx.x,
                            gridDim.x * blockDim.x, blockIdx.x == 0);
}

// ---------------------------------------------------------------------------
// Unpacks the sweep state into the caller's velocities; with integrate the
// positions (and 2D orientations) follow Eq. 2 and the walls move.
// ---------------------------------------------------------------------------
template <int DIM, typename T>
__global__ void k_unpack(CdGeom g, CdWork w, double* __restrict__ pos, double* __restrict__ vel,
                         double* __restrict__ omega, double* __restrict__ theta, int integrate)
{
    if (w.ctrl->skip) return;
    typedef typename Vec<T>::V4 T4;
    const T4* V = (const T4*)w.V;
    const CdState io{pos, vel, omega, theta, integrate};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.n; i += gridDim.x * blockDim.x) {
        if constexpr (DIM == 2) unpack_particle<2, T>(g, io, i, V[i], V[i]);
        else unpack_particle<3, T>(g, io, i, V[2 * i], V[2 * i + 1]);
    }
    if (g.dyn_walls && blockIdx.x == 0 && threadIdx.x == 0) unpack_walls<DIM, T>(g, w);
    if (integrate) {
        if (g.dyn_walls) __syncthreads();   // block 0 moves the walls after their velocities are written
        for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < g.npk; b += gridDim.x * blockDim.x)
            move_walls<DIM>(g, w, b);
    }
}

// Loads this thread's first record of colour k (if it has one) into nxt.
template <int DIM, typename T, bool VIEWS = false>
__device__ __forceinline__ void prefetch_first(const CdGeom& g, const CdWork& w, const int* s_off, int k,
                                               Rec<DIM, T>& nxt)
{
    const CdSpan sq = cd_colour_span(s_off[k], s_off[k + 1]);
    if (sq.p < sq.end) load_rec<DIM, T, VIEWS>(g, w, sq.p, nxt);
}

// Loads this thread's first record of phase k: of the colour class, or of
// this block's first list of the merged phase.
template <int DIM, typename T, int MODE>
__device__ __forceinline__ void prefetch_any(const CdGeom& g, const CdWork& w, const int* s_off, int k,
                                             Rec<DIM, T>& nxt, const MgInfo& mg)
{
    if constexpr (MODE == CD_SWEEP_MERGE) {
        if (mg.on && k == mg.klast) {
            // item q = threadIdx.x of the block's lists taken in turn
            int q = (int)threadIdx.x;
            for (int m = 0; m < mg.M; ++m) {
                const int cnt = mg.lst[2 * m + 1] - mg.lst[2 * m];
                if (q < cnt) {
                    load_rec<DIM, T>(g, w, w.mg_list[mg.lst[2 * m] + q], nxt);
                    break;
                }
                q -= cnt;
            }
            return;
        }
    }
    prefetch_first<DIM, T, MODE == CD_SWEEP_DOMAINS>(g, w, s_off, k, nxt);
}

// One colour phase for this thread: its first contact's record was loaded
// into `nxt` before the barrier (if it has one); the rest are loaded inline.
// Afterwards `nxt` holds the first record of colour `knext` (prefetch).
// `pend` carries (P_n, P_t) of the thread's last update whose magnitude is
// not yet in acc[0] (zeros if none) from phase to phase; the caller adds it
// before the block sum at the end of a pass.
template <int DIM, typename T, int MODE>
__device__ __forceinline__ void colour_phase(const CdGeom& g, const CdWork& w, const int* s_off, int k, int knext,
                                             int tid, int stride, Rec<DIM, T>& nxt, bool apply_only, int crit,
                                             double alpha, double ravg_prev, double (&acc)[3], double2& pend,
                                             const MgInfo& mg, bool skip_first = false)
{
    constexpr bool MIXED = (MODE == CD_SWEEP_MIXED);
    constexpr bool VIEWS = (MODE == CD_SWEEP_DOMAINS);
    // FP64 2D only: FP32 takes its square root on the fast pipe, and in 3D the
    // extra live value spills
    constexpr bool DEFER = (DIM == 2) && std::is_same<T, double>::value;
    if constexpr (MODE == CD_SWEEP_MERGE) {
        if (mg.on && k == mg.klast) {
            // the chains' contacts of colour K-M, a block barrier, those of K-M+1, ...
            const int t = (int)threadIdx.x, bd = (int)blockDim.x;
            int base = 0;   // items of the earlier lists
            for (int m = 0; m < mg.M; ++m) {
                const int l0 = mg.lst[2 * m], cnt = mg.lst[2 * m + 1] - l0;
                int q0 = t;
                if (q0 < base) q0 += ((base - q0 + bd - 1) / bd) * bd;   // this thread's first item of list m
                for (int q = q0; q < base + cnt; q += bd) {
                    const int p = w.mg_list[l0 + (q - base)];
                    UpdOut o;
                    if (q == t) {
                        o = apply_rec<DIM, T, false, DEFER>(g, w, p, nxt, apply_only, crit, alpha, ravg_prev, pend);
                    } else {
                        Rec<DIM, T> r;
                        load_rec<DIM, T>(g, w, p, r);
                        o = apply_rec<DIM, T, false, DEFER>(g, w, p, r, apply_only, crit, alpha, ravg_prev, pend);
                    }
                    acc[0] += o.pabs;
                    if (DEFER) pend = make_double2(o.pn, o.pt);
                    if (crit == CD_CONV_LOCAL) { acc[1] += (double)o.rel_ok; acc[2] += (double)o.bad; }
                }
                base += cnt;
                if (m + 1 < mg.M) __syncthreads();
            }
            if (knext >= 0) prefetch_any<DIM, T, MODE>(g, w, s_off, knext, nxt, mg);
            return;
        }
    }
    const CdSpan sp = cd_colour_span(s_off[k], s_off[k + 1]);
    const int end = sp.end;
    int p = sp.p;
    const bool mixed = MIXED && !apply_only;   // parallel contacts were done in their own phase
    if (p < end) {
        // skip_first: this thread's first update of the phase was staged and
        // stored before the phase (the first colour of a sweep, see k_sweep)
        if (!skip_first && !(mixed && cd_is_parallel(g.par_p, g.seed, cd_key(nxt.ab.x, nxt.ab.y), mg.draw))) {
            UpdOut o = apply_rec<DIM, T, VIEWS, DEFER>(g, w, p, nxt, apply_only, crit, alpha, ravg_prev, pend);
            acc[0] += o.pabs;
            if (DEFER) pend = make_double2(o.pn, o.pt);
            if (crit == CD_CONV_LOCAL) { acc[1] += (double)o.rel_ok; acc[2] += (double)o.bad; }
        }
        for (p += blockDim.x; p < end; p += blockDim.x) {
            Rec<DIM, T> r;
            load_rec<DIM, T, VIEWS>(g, w, p, r);
            if (mixed && cd_is_parallel(g.par_p, g.seed, cd_key(r.ab.x, r.ab.y), mg.draw)) continue;
            UpdOut o = apply_rec<DIM, T, VIEWS, DEFER>(g, w, p, r, apply_only, crit, alpha, ravg_prev, pend);
            acc[0] += o.pabs;
            if (DEFER) pend = make_double2(o.pn, o.pt);
            if (crit == CD_CONV_LOCAL) { acc[1] += (double)o.rel_ok; acc[2] += (double)o.bad; }
        }
    }
    if (knext >= 0) prefetch_any<DIM, T, MODE>(g, w, s_off, knext, nxt, mg);
    (void)tid; (void)stride;
}

// ---------------------------------------------------------------------------
// Mixed update (Sec. 2.3).  Parallel contacts compute their new impulse from
// the velocities at the start of the sweep (no velocity change yet) and keep
// the change; after the sequential colours each particle adds the changes of
// its parallel contacts in ascending key order.
// ---------------------------------------------------------------------------
template <int DIM, typename T>
__device__ __forceinline__ UpdOut par_compute(const CdGeom& g, const CdWork& w, int p, const Rec<DIM, T>& r, int crit,
                                              double alpha, double ravg_prev)
{
    typedef typename Vec<T>::V4 T4;
    typedef typename Vec<T>::V2 T2;
    const T4* V = (const T4*)w.V;
    const bool wall = r.ab.y >= g.n;
    const int c = w.perm[p];
    UpdOut o;
    Rec<DIM, T> rs = r;
    if constexpr (sizeof(T) == 8) load_static<DIM, T>(g, w, rs);
    if constexpr (DIM == 2) {
        T4 va = V[r.ab.x], vb;
        if (!wall) vb = V[r.ab.y];
        else wall_vel2<T>(g, w, r.ab.y, vb);
        T2 Pnew;
        o = core2d<T>(g, rs, va, vb, wall, false, crit, alpha, ravg_prev, Pnew);
        ((T2*)w.c_P)[p] = Pnew;
        w.c_dpar[2 * c] = (double)(Pnew.x - r.P.x);
        w.c_dpar[2 * c + 1] = (double)(Pnew.y - r.P.y);
    } else {
        T4 va = V[2 * r.ab.x], wa = V[2 * r.ab.x + 1], vb, wb;
        if (!wall) { vb = V[2 * r.ab.y]; wb = V[2 * r.ab.y + 1]; }
        else wall_vel3<T>(g, w, r.ab.y, vb, wb);
        T4 Pnew;
        o = core3d<T>(g, rs, va, wa, vb, wb, wall, false, crit, alpha, ravg_prev, Pnew);
        ((T4*)w.c_P)[p] = Pnew;
        w.c_dpar[4 * c] = (double)(Pnew.x - r.P.x);
        w.c_dpar[4 * c + 1] = (double)(Pnew.y - r.P.y);
        w.c_dpar[4 * c + 2] = (double)(Pnew.z - r.P.z);
        w.c_dpar[4 * c + 3] = (double)(Pnew.w - r.P.w);
    }
    return o;
}

template <int DIM, typename T>
__device__ __forceinline__ void par_apply(const CdGeom& g, const CdWork& w, int tid, int stride, long long draw)
{
    typedef typename Vec<T>::V4 T4;
    T4* V = (T4*)w.V;
    const T4* S = (const T4*)w.S;
    for (int i = tid; i < g.n; i += stride) {
        const int e = w.p2c_off[i + 1];
        bool any = false;
        T4 v, om;
        const T4 si = S[i];
        for (int q = w.p2c_off[i]; q < e; ++q) {
            const int c = w.p2c[q];
            const int2 ab = w.pairs[c];
            if (!cd_is_parallel(g.par_p, g.seed, cd_key(ab.x, ab.y), draw)) continue;
            if (!any) {
                any = true;
                if (DIM == 2) v = V[i];
                else { v = V[2 * i]; om = V[2 * i + 1]; }
            }
            const T sign = (ab.x == i) ? (T)-1 : (T)1;
            const T nx = (T)w.nrm[3 * c], ny = (T)w.nrm[3 * c + 1], nz = (T)w.nrm[3 * c + 2];
            if (DIM == 2) {
                const T dPn = (T)w.c_dpar[2 * c], dPt = (T)w.c_dpar[2 * c + 1];
                const T dx = dPn * nx - dPt * ny, dy = dPn * ny + dPt * nx;
                v.x += sign * si.x * dx; v.y += sign * si.x * dy;
                v.z -= si.z * dPt;
            } else {
                const T dPn = (T)w.c_dpar[4 * c];
                const T dx = dPn * nx + (T)w.c_dpar[4 * c + 1];
                const T dy = dPn * ny + (T)w.c_dpar[4 * c + 2];
                const T dz = dPn * nz + (T)w.c_dpar[4 * c + 3];
                const T cx = ny * dz - nz * dy, cy = nz * dx - nx * dz, cz = nx * dy - ny * dx;
                v.x += sign * si.x * dx; v.y += sign * si.x * dy; v.z += sign * si.x * dz;
                om.x -= si.z * cx; om.y -= si.z * cy; om.z -= si.z * cz;
            }
        }
        if (any) {
            if (DIM == 2) store_xyz_plain<T>(V + i, v);
            else { store_xyz_plain<T>(V + 2 * i, v); V[2 * i + 1] = om; }
        }
    }
}

// ---------------------------------------------------------------------------
// Domain-wise update (Sec. 3.1).  Each contact updates the velocity records
// of its domain (c_vab).  Before the first pass every view record takes its
// particle's velocity; after every pass (the starting impulses, then each
// sweep) a particle with views gets v0 + (v_home - v0) + sum over its views
// in ascending domain order of (v_view - v0), v0 being the velocity of the
// pass start, and every view starts the next pass from that sum.
// ---------------------------------------------------------------------------
template <int DIM, typename T>
__device__ __forceinline__ void dom_init(const CdGeom& g, const CdWork& w, int tid, int stride)
{
    typedef typename Vec<T>::V4 T4;
    constexpr int RW = (DIM == 2) ? 1 : 2;   // records per body
    T4* V = (T4*)w.V;
    T4* V0 = (T4*)w.V0;
    const int nv = w.view_off[g.n], base = cd_view_base(g);
    for (int q = tid; q < nv; q += stride) {
        const int i = w.view_owner[q];
#pragma unroll
        for (int h = 0; h < RW; ++h) {
            const T4 x = V[RW * i + h];
            V[RW * (base + q) + h] = x;
            V0[RW * q + h] = x;
        }
    }
}

template <int DIM, typename T>
__device__ __forceinline__ void dom_combine(const CdGeom& g, const CdWork& w, int tid, int stride)
{
    typedef typename Vec<T>::V4 T4;
    constexpr int RW = (DIM == 2) ? 1 : 2;
    T4* V = (T4*)w.V;
    T4* V0 = (T4*)w.V0;
    const int nv = w.view_off[g.n], base = cd_view_base(g);
    for (int q = tid; q < nv; q += stride) {
        const int i = w.view_owner[q];
        if (q != w.view_off[i]) continue;   // one thread per particle: its first view
        const int e = w.view_off[i + 1];
#pragma unroll
        for (int h = 0; h < RW; ++h) {
            const T4 s0 = V0[RW * q + h];
            T4 x = V[RW * i + h];
            T sx = s0.x + (x.x - s0.x), sy = s0.y + (x.y - s0.y), sz = s0.z + (x.z - s0.z);
            for (int u = q; u < e; ++u) {
                const T4 a = V[RW * (base + u) + h];
                sx = sx + (a.x - s0.x);
                sy = sy + (a.y - s0.y);
                sz = sz + (a.z - s0.z);
            }
            x.x = sx; x.y = sy; x.z = sz;
            V[RW * i + h] = x;
            for (int u = q; u < e; ++u) {
                V[RW * (base + u) + h] = x;
                V0[RW * u + h] = x;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// The persistent sweep kernel
// ---------------------------------------------------------------------------
// MODE: CD_SWEEP_PLAIN, CD_SWEEP_MIXED (the mixed update of Sec. 2.3,
// params.parallel_p > 0) or CD_SWEEP_DOMAINS (the domain-wise update of
// Sec. 3.1, params.domains); each variant carries only its own code.
template <int DIM, typename T, int MODE>
__global__ void __launch_bounds__(CD_SWEEP_THREADS, 1)
k_sweep(CdGeom g, CdWork w, int crit, double alpha, int max_sweeps)
{
    constexpr bool MIXED = (MODE == CD_SWEEP_MIXED);
    constexpr bool VIEWS = (MODE == CD_SWEEP_DOMAINS);
    __shared__ int s_off[CD_KMAX + 1];
    __shared__ double s_red[CD_SWEEP_THREADS / 32][3];
    __shared__ double s_bc;
    CdCtrl* ctrl = w.ctrl;
    if (ctrl->skip) return;
    const int nc = ctrl->nc;
    int K = ctrl->ncolours;
    const int nb = gridDim.x;
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int stride = gridDim.x * blockDim.x;
    unsigned long long epoch = 0;
    for (int k = threadIdx.x; k <= CD_KMAX; k += blockDim.x) s_off[k] = w.colour_off[k];
    MgInfo mg;
    mg.on = 0; mg.klast = -1; mg.M = 0; mg.lst = nullptr; mg.draw = -1;
    __shared__ int s_mgl[2 * CD_MG_MAXC];
    if constexpr (MODE == CD_SWEEP_MERGE) {
        const int M = ctrl->merge;
        if (M >= 2 && M <= CD_MG_MAXC && nb == g.merge_blocks) {
            // the M last colours run as one phase (lists built for this grid)
            mg.on = 1;
            mg.M = M;
            K -= M - 1;
            mg.klast = K - 1;
            const int b = blockIdx.x;
            if (threadIdx.x < 2 * M) {
                const int m = threadIdx.x >> 1;
                s_mgl[threadIdx.x] = w.mg_boff[m * nb + b + (threadIdx.x & 1)];
            }
            mg.lst = s_mgl;
        }
    }
    __syncthreads();

    int sweeps = 0, converged = (nc == 0);
    double resid = 0.0, ravg = 0.0, ravg_prev = 0.0;
    if (nc > 0) {
        if constexpr (VIEWS) {
            dom_init<DIM, T>(g, w, tid, stride);
            if (!cd_grid_sync(ctrl, nb, epoch)) return;
        }
        Rec<DIM, T> nxt;
        prefetch_any<DIM, T, MODE>(g, w, s_off, 0, nxt, mg);
        // starting impulses, colour by colour
        double acc[3] = {0.0, 0.0, 0.0};
        double2 pend = make_double2(0.0, 0.0);   // this thread's last impulse not yet in the residual sum
        for (int k = 0; k < K; ++k) {
            colour_phase<DIM, T, MODE>(g, w, s_off, k, (k + 1 < K) ? k + 1 : 0, tid, stride, nxt, true, crit, alpha,
                                       0.0, acc, pend, mg);
            if (k == K - 1) {
                acc[0] += abs_of_pair(pend.x, pend.y);
                pend = make_double2(0.0, 0.0);
                block_sum<3>(acc, s_red, 1);
                if (threadIdx.x == 0) w.partials[blockIdx.x] = acc[0];
            }
            if (!cd_grid_sync(ctrl, nb, epoch)) return;
        }
        if constexpr (VIEWS) {
            dom_combine<DIM, T>(g, w, tid, stride);
            if (!cd_grid_sync(ctrl, nb, epoch)) return;
        }
        ravg_prev = grid_total(w.partials, nb, &s_bc) / (double)nc;
        ravg = ravg_prev;

        // 2D plain and merged schedules under the global tests: while the last
        // warp of each block runs the convergence test of sweep j, the other
        // threads compute their first update of sweep j + 1 (colour 0, its
        // record prefetched) into registers and store it only if the test
        // says continue.  The same updates in the same order: bits unchanged.
        constexpr bool SPEC_OK = (DIM == 2) && !MIXED && !VIEWS;
        const bool spec_on = SPEC_OK && crit != CD_CONV_LOCAL && !(mg.on && mg.klast == 0);
        bool spec_done = false;   // this thread's first colour-0 update of the coming sweep is stored
        double carry = 0.0;       // its residual term (the first term of the sweep's sum)
        while (!converged && sweeps < max_sweeps) {
            const int buf = (sweeps & 1) ? 0 : 1;   // alternate with the buffer of the previous sweep
            double* part = w.partials + (size_t)buf * 3 * nb;
            double a3[3] = {carry, 0.0, 0.0};
            carry = 0.0;
            const bool mixed = MIXED;
            if (MIXED && g.par_redraw) mg.draw = sweeps;   // this iteration step's parallel subset
            if (mixed) {
                for (int p = tid; p < nc; p += stride) {
                    Rec<DIM, T> r;
                    load_rec<DIM, T>(g, w, p, r);
                    if (!cd_is_parallel(g.par_p, g.seed, cd_key(r.ab.x, r.ab.y), mg.draw)) continue;
                    UpdOut o = par_compute<DIM, T>(g, w, p, r, crit, alpha, ravg_prev);
                    a3[0] += o.pabs;
                    if (crit == CD_CONV_LOCAL) { a3[1] += (double)o.rel_ok; a3[2] += (double)o.bad; }
                }
                if (!cd_grid_sync(ctrl, nb, epoch)) return;
                // the prefetched record of colour 0 may belong to a parallel contact whose
                // impulse just changed: reload it
                const CdSpan s0 = cd_colour_span(s_off[0], s_off[1]);
                if (s0.p < s0.end) load_rec<DIM, T>(g, w, s0.p, nxt);
            }
            for (int k = 0; k < K; ++k) {
                // no prefetch inside the phase: it is issued after the barrier arrival
                // below, so that the arriving thread's fence does not wait for it
                colour_phase<DIM, T, MODE>(g, w, s_off, k, -1, tid, stride, nxt, false, crit, alpha, ravg_prev, a3,
                                           pend, mg, k == 0 && spec_done);
                if (k == K - 1) {
                    // (a thread without a pending impulse adds nothing: skip the FP64 work)
                    if ((__double_as_longlong(pend.x) | __double_as_longlong(pend.y)) != 0)
                        a3[0] += abs_of_pair(pend.x, pend.y);
                    pend = make_double2(0.0, 0.0);
                }
                if (mixed && k == K - 1) {
                    if (!cd_grid_sync(ctrl, nb, epoch)) return;
                    par_apply<DIM, T>(g, w, tid, stride, mg.draw);
                }
                if (k == K - 1) {
                    block_sum<3>(a3, s_red, test_values(crit));
                    if (threadIdx.x == 0) {
                        part[blockIdx.x] = a3[0];
                        part[nb + blockIdx.x] = a3[1];
                        part[2 * nb + blockIdx.x] = a3[2];
                    }
                }
                const unsigned old = cd_grid_arrive(ctrl, nb);
                if (!mixed || k + 1 < K) prefetch_any<DIM, T, MODE>(g, w, s_off, (k + 1 < K) ? k + 1 : 0, nxt, mg);
                if (!cd_grid_wait(ctrl, old, epoch)) return;
            }
            if constexpr (VIEWS) {
                dom_combine<DIM, T>(g, w, tid, stride);
                if (!cd_grid_sync(ctrl, nb, epoch)) return;
            }
            ++sweeps;
            spec_done = false;
            if constexpr (SPEC_OK) {
                constexpr bool DEFER = std::is_same<T, double>::value;
                Staged2<T> st;
                bool staged = false;
                if (spec_on && sweeps < max_sweeps) {
                    const CdSpan s0 = cd_colour_span(s_off[0], s_off[1]);
                    if (s0.p < s0.end) {
                        // pend is (0, 0) here (the last phase added it to the sum), so
                        // the staged update's own residual term is 0 under DEFER
                        (void)stage2d<T, false, DEFER>(g, w, s0.p, nxt, false, crit, alpha, ravg_prev, pend, st);
                        staged = true;
                    }
                }
                sweep_test(part, nb, nc, crit, alpha, ravg_prev, ravg, resid, converged, s_red[0]);
                if (staged && !converged) {
                    commit2d<T>(w, st);
                    spec_done = true;
                    if constexpr (DEFER) {
                        pend = make_double2((double)st.P.x, (double)st.P.y);   // its |P| joins the sum later
                    } else {
                        // |P| of the update, as core2d takes it in this precision
                        carry = abs_of_sq<T>((double)fma_of<T>(st.P.y, st.P.y, mul_of<T>(st.P.x, st.P.x)));
                    }
                }
            } else {
                sweep_test(part, nb, nc, crit, alpha, ravg_prev, ravg, resid, converged, s_red[0]);
            }
            ravg_prev = ravg;
        }
    }

    finish_solve<DIM, T>(g, w, nc, nb, tid, stride, epoch, sweeps, converged, resid, ravg, s_red);
}

// ---------------------------------------------------------------------------
// Batched systems: independent packings share the colour phases (so each
// grid barrier is amortised over all of them) but each has its own
// convergence test.  After a sweep every block reduces |P| over the
// contiguous key-order contact range of the packings it owns (fixed order:
// deterministic), decides convergence, and a converged packing's contacts are
// skipped from the next sweep on, exactly as if it were solved alone.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void pk_reduce(const CdGeom& g, const CdWork& w, int sweep, int crit, double alpha,
                                          int* act_slot, int* act_c_slot, double (*s_red)[3])
{
    for (int b = blockIdx.x; b < g.npk; b += gridDim.x) {
        double* st = w.pk_stats + CD_PKSTATS * b;
        if (sweep >= 0 && cd_ld_volatile_int(&w.pk_done[b])) continue;
        const int c0 = w.pk_coff[b], c1 = w.pk_coff[b + 1];
        double a3[3] = {0.0, 0.0, 0.0};
        for (int c = c0 + threadIdx.x; c < c1; c += blockDim.x) {
            a3[0] += w.c_abs[c];
            if (crit == CD_CONV_LOCAL && sweep >= 0) {
                int f = w.c_flag[c];
                a3[1] += (double)(f & 1);
                a3[2] += (double)((f >> 1) & 1);
            }
        }
        block_sum<3>(a3, s_red, (crit == CD_CONV_LOCAL && sweep >= 0) ? 3 : 1);
        if (threadIdx.x == 0) {
            const int ncb = c1 - c0;
            const double R = (ncb > 0) ? a3[0] / (double)ncb : 0.0;
            if (sweep < 0) {
                st[PKS_SWEEPS] = 0.0;
                st[PKS_CONV] = (ncb == 0) ? 1.0 : 0.0;
                st[PKS_RESID] = 0.0;
                st[PKS_RAVG] = R;
                st[PKS_RPREV] = R;
                st[PKS_NC] = (double)ncb;
                w.pk_done[b] = (ncb == 0) ? 1 : 0;
            } else {
                const double Rp = st[PKS_RPREV], den = R + Rp;
                double resid;
                int conv;
                if (crit == CD_CONV_GLOBAL_REL) {
                    resid = (den > 0.0) ? fabs(R - Rp) / den : (den == 0.0 ? 0.0 : den);
                    conv = resid < alpha;
                } else if (crit == CD_CONV_GLOBAL_SQ) {
                    double q = (den > 0.0) ? (R - Rp) / den : (den == 0.0 ? 0.0 : den);
                    resid = q * q;
                    conv = resid < alpha;
                } else if (crit == CD_CONV_LOCAL) {
                    resid = (ncb > 0) ? (double)(ncb - (long long)a3[1]) / (double)ncb : 0.0;
                    conv = (10.0 * a3[1] >= 9.0 * (double)ncb) && a3[2] == 0.0;
                } else {
                    resid = (den > 0.0) ? fabs(R - Rp) / den : (den == 0.0 ? 0.0 : den);
                    conv = 0;
                }
                st[PKS_SWEEPS] = (double)(sweep + 1);
                st[PKS_RESID] = resid;
                st[PKS_RAVG] = R;
                st[PKS_RPREV] = R;
                if (conv) {
                    st[PKS_CONV] = 1.0;
                    w.pk_done[b] = 1;
                } else {
                    atomicAdd(act_slot, 1);
                    atomicAdd(act_c_slot, ncb);
                }
            }
        }
        __syncthreads();
    }
}

// Exclusive scan of a 0/1 flag over the block (ballot per warp, warp totals in
// shared memory); returns the flags before this thread, *total the block's sum.
__device__ __forceinline__ int block_excl_scan01(int f, int* s_warp, int* total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const unsigned m = __ballot_sync(0xffffffffu, f);
    const int in_warp = __popc(m & ((1u << lane) - 1u));
    if (lane == 0) s_warp[wid] = __popc(m);
    __syncthreads();
    int before = 0, tot = 0;
    for (int q = 0; q < nw; ++q) {
        const int c = s_warp[q];
        if (q < wid) before += c;
        tot += c;
    }
    __syncthreads();
    *total = tot;
    return before + in_warp;
}

// Drops the contacts of converged packings from the colour-order arrays: a
// stable partition into the second set of arrays, copied back to the front of
// the first, so that later sweeps spread only the active contacts over the
// grid.  A dropped contact's final impulse goes back to key order here.
// Colour order and the updates themselves are unchanged, so results are
// identical.  Returns the new number of positions (same in every block).
template <int DIM, typename T>
__device__ __forceinline__ int compact_batch(const CdGeom& g, const CdWork& w, int nact, int K, int* s_off,
                                             unsigned long long& epoch, bool& ok)
{
    typedef typename Vec<T>::V4 T4;
    typedef typename Vec<T>::V2 T2;
    __shared__ int s_warp[CD_SWEEP_THREADS / 32];
    __shared__ int s_base;
    CdCtrl* ctrl = w.ctrl;
    const int nb = gridDim.x;
    const int chunk = (nact + nb - 1) / nb;
    const int lo = min((int)blockIdx.x * chunk, nact), hi = min(lo + chunk, nact);
    auto keep = [&](int p) { return cd_ld_volatile_int(&w.pk_done[w.pack_of[w.c_ab[p].x]]) == 0; };
    int cnt = 0;
    for (int p = lo + (int)threadIdx.x; p < hi; p += blockDim.x) cnt += keep(p) ? 1 : 0;
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int q = 0; q < (int)(blockDim.x >> 5); ++q) t += s_warp[q];
        w.cmp_blk[blockIdx.x] = t;
    }
    if (!cd_grid_sync(ctrl, nb, epoch)) { ok = false; return nact; }
    if (threadIdx.x == 0) {
        int b0 = 0, tot = 0;
        for (int q = 0; q < nb; ++q) {
            const int c = cd_ld_volatile_int(&w.cmp_blk[q]);
            if (q < (int)blockIdx.x) b0 += c;
            tot += c;
        }
        s_base = b0;
        if (blockIdx.x == 0)
            for (int k = 0; k <= K; ++k)
                if (s_off[k] == nact) w.cmp_off[k] = tot;
    }
    __syncthreads();
    int running = s_base;
    const int pw = (DIM == 2) ? 2 : 4;
    for (int t0 = lo; t0 < hi; t0 += blockDim.x) {
        const int p = t0 + (int)threadIdx.x;
        const int f = (p < hi) && keep(p);
        int tile_tot;
        const int ex = block_excl_scan01(f, s_warp, &tile_tot);
        if (p < hi) {
            for (int k = 0; k <= K; ++k)
                if (s_off[k] == p) w.cmp_off[k] = running + ex;
            if (f) {
                const int q = running + ex;
                w.c_ab2[q] = w.c_ab[p];
                ((T4*)w.c_geo2)[q] = ((const T4*)w.c_geo)[p];
                if constexpr (DIM == 2) {
                    ((T*)w.c_m2)[q] = ((const T*)w.c_m)[p];
                    ((T2*)w.c_P2)[q] = ((const T2*)w.c_P)[p];
                } else {
                    ((T2*)w.c_m2)[q] = ((const T2*)w.c_m)[p];
                    ((T4*)w.c_P2)[q] = ((const T4*)w.c_P)[p];
                }
                w.perm2[q] = w.perm[p];
            } else {
                const int c = w.perm[p];
                if constexpr (DIM == 2) {
                    const T2 P = ((const T2*)w.c_P)[p];
                    w.Pk[pw * c] = (double)P.x;
                    w.Pk[pw * c + 1] = (double)P.y;
                } else {
                    const T4 P = ((const T4*)w.c_P)[p];
                    w.Pk[pw * c] = (double)P.x; w.Pk[pw * c + 1] = (double)P.y;
                    w.Pk[pw * c + 2] = (double)P.z; w.Pk[pw * c + 3] = (double)P.w;
                }
            }
        }
        running += tile_tot;
    }
    if (!cd_grid_sync(ctrl, nb, epoch)) { ok = false; return nact; }
    int tot = 0;
    for (int q = 0; q < nb; ++q) tot += cd_ld_volatile_int(&w.cmp_blk[q]);
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < tot; q += gridDim.x * blockDim.x) {
        w.c_ab[q] = w.c_ab2[q];
        ((T4*)w.c_geo)[q] = ((const T4*)w.c_geo2)[q];
        if constexpr (DIM == 2) {
            ((T*)w.c_m)[q] = ((const T*)w.c_m2)[q];
            ((T2*)w.c_P)[q] = ((const T2*)w.c_P2)[q];
        } else {
            ((T2*)w.c_m)[q] = ((const T2*)w.c_m2)[q];
            ((T4*)w.c_P)[q] = ((const T4*)w.c_P2)[q];
        }
        w.perm[q] = w.perm2[q];
    }
    if (!cd_grid_sync(ctrl, nb, epoch)) { ok = false; return nact; }
    for (int k = threadIdx.x; k <= K; k += blockDim.x) s_off[k] = cd_ld_volatile_int(&w.cmp_off[k]);
    __syncthreads();
    return tot;
}

template <int DIM, typename T>
__global__ void __launch_bounds__(CD_SWEEP_THREADS, 1)
k_sweep_batch(CdGeom g, CdWork w, int crit, double alpha, int max_sweeps)
{
    __shared__ int s_off[CD_KMAX + 1];
    __shared__ double s_red[CD_SWEEP_THREADS / 32][3];
    CdCtrl* ctrl = w.ctrl;
    if (ctrl->skip || (g.flow && !w.fl_plan->barriers)) return;   // (solved by dataflow)
    const int nc = ctrl->nc;
    const int K = ctrl->ncolours;
    const int nb = gridDim.x;
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int stride = gridDim.x * blockDim.x;
    unsigned long long epoch = 0;
    for (int k = threadIdx.x; k <= CD_KMAX; k += blockDim.x) s_off[k] = w.colour_off[k];
    if (tid == 0)
        for (int q = 0; q < 6; ++q) w.act_cnt[q] = 0;
    __syncthreads();
    int nact = nc;   // positions still in the colour-order arrays

    // starting impulses, colour by colour
    for (int k = 0; k < K; ++k) {
        const CdSpan sp = cd_colour_span(s_off[k], s_off[k + 1]);
        for (int p = sp.p; p < sp.end; p += blockDim.x) {
            Rec<DIM, T> r;
            load_rec<DIM, T>(g, w, p, r);
            UpdOut o = apply_rec<DIM, T>(g, w, p, r, true, crit, alpha, 0.0);
            w.c_abs[w.perm[p]] = o.pabs;
        }
        if (!cd_grid_sync(ctrl, nb, epoch)) return;
    }
    pk_reduce(g, w, -1, crit, alpha, nullptr, nullptr, s_red);
    if (!cd_grid_sync(ctrl, nb, epoch)) return;

    for (int sweep = 0; sweep < max_sweeps && nc > 0; ++sweep) {
        if (tid == 0) { w.act_cnt[(sweep + 1) % 3] = 0; w.act_cnt[3 + (sweep + 1) % 3] = 0; }
        for (int k = 0; k < K; ++k) {
            const CdSpan sp = cd_colour_span(s_off[k], s_off[k + 1]);
            for (int p = sp.p; p < sp.end; p += blockDim.x) {
                Rec<DIM, T> r;
                load_rec<DIM, T>(g, w, p, r);
                if (w.pk_done[r.pk]) continue;
                const double rprev = (crit == CD_CONV_LOCAL) ? w.pk_stats[CD_PKSTATS * r.pk + PKS_RPREV] : 0.0;
                UpdOut o = apply_rec<DIM, T>(g, w, p, r, false, crit, alpha, rprev);
                const int c = w.perm[p];
                w.c_abs[c] = o.pabs;
                w.c_flag[c] = o.rel_ok | (o.bad << 1);
            }
            if (!cd_grid_sync(ctrl, nb, epoch)) return;
        }
        pk_reduce(g, w, sweep, crit, alpha, &w.act_cnt[sweep % 3], &w.act_cnt[3 + sweep % 3], s_red);
        if (!cd_grid_sync(ctrl, nb, epoch)) return;
        if (cd_ld_volatile_int(&w.act_cnt[sweep % 3]) == 0) break;
        // once a third of the positions belong to converged packings, drop them
        const int live = cd_ld_volatile_int(&w.act_cnt[3 + sweep % 3]);
        if (3 * (nact - live) >= nact && sweep + 1 < max_sweeps) {
            bool ok = true;
            nact = compact_batch<DIM, T>(g, w, nact, K, s_off, epoch, ok);
            if (!ok) return;
        }
    }

    // impulses back to key order (those of dropped contacts were written when dropped)
    typedef typename Vec<T>::V4 T4;
    typedef typename Vec<T>::V2 T2;
    for (int p = tid; p < nact; p += stride) {
        int c = w.perm[p];
        if (DIM == 2) {
            T2 P = ((const T2*)w.c_P)[p];
            w.Pk[2 * c] = (double)P.x;
            w.Pk[2 * c + 1] = (double)P.y;
        } else {
            T4 P = ((const T4*)w.c_P)[p];
            w.Pk[4 * c] = (double)P.x; w.Pk[4 * c + 1] = (double)P.y;
            w.Pk[4 * c + 2] = (double)P.z; w.Pk[4 * c + 3] = (double)P.w;
        }
    }
    if (!cd_grid_sync(ctrl, nb, epoch)) return;
    // per-packing wall forces and the call's totals
    const int pw = (DIM == 2) ? 2 : 4;
    for (int b = blockIdx.x; b < g.npk; b += gridDim.x) {
        const int c0 = w.pk_coff[b], c1 = w.pk_coff[b + 1];
        double lo3[3] = {0.0, 0.0, 0.0}, hi3[3] = {0.0, 0.0, 0.0};
        for (int c = c0 + threadIdx.x; c < c1; c += blockDim.x) {
            int bb = w.pairs[c].y;
            if (bb < g.n) continue;
            int k = (bb - g.n) % 6;
            double pn = w.Pk[pw * c];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                if (q == k) lo3[q] += pn;
                if (q + 3 == k) hi3[q] += pn;
            }
        }
        block_sum<3>(lo3, s_red);
        block_sum<3>(hi3, s_red);
        if (threadIdx.x == 0) {
            double* st = w.pk_stats + CD_PKSTATS * b;
            for (int q = 0; q < 3; ++q) {
                st[PKS_WF0 + q] = lo3[q] / g.dt;
                st[PKS_WF0 + 3 + q] = hi3[q] / g.dt;
            }
            const long long sw = (long long)st[PKS_SWEEPS];
            atomicAdd((unsigned long long*)&ctrl->total_updates, (unsigned long long)(sw * (long long)(c1 - c0)));
            atomicMax((unsigned long long*)&ctrl->max_sweeps_step, (unsigned long long)sw);
            if (st[PKS_CONV] == 0.0) atomicAdd((unsigned long long*)&ctrl->n_not_conv, 1ULL);
            if (b == 0) {
                for (int q = 0; q < 6; ++q) ctrl->wall_force[q] = st[PKS_WF0 + q];
                ctrl->r_avg = st[PKS_RAVG];
                ctrl->residual = st[PKS_RESID];
            }
        }
        __syncthreads();
    }
    if (!cd_grid_sync(ctrl, nb, epoch)) return;
    if (tid == 0) {
        ctrl->steps_done += 1;
        long long tot = 0, mx = 0, open = 0;
        for (int b = 0; b < g.npk; ++b) {
            const long long sw = (long long)w.pk_stats[CD_PKSTATS * b + PKS_SWEEPS];
            tot += sw;
            if (sw > mx) mx = sw;
            if (w.pk_stats[CD_PKSTATS * b + PKS_CONV] == 0.0) ++open;
        }
        ctrl->total_sweeps += tot;
        ctrl->sweeps = mx;
        ctrl->converged = (open == 0);
    }
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
static int grid_n(int n)
{
    int g = (n + CD_BLOCK - 1) / CD_BLOCK;
    return g < 1 ? 1 : (g > 4096 ? 4096 : g);
}

cudaError_t cd_launch_static(const CdGeom& g, const CdWork& w, const double* radius, const double* inv_m,
                             const double* inv_I, int precision, cudaStream_t s, int* nl)
{
    if (precision == CD_FP64)
        k_static<double><<<grid_n(g.n), CD_BLOCK, 0, s>>>(g, g.n, g.rotations, radius, inv_m, inv_I, (Vec<double>::V4*)w.S);
    else
        k_static<float><<<grid_n(g.n), CD_BLOCK, 0, s>>>(g, g.n, g.rotations, radius, inv_m, inv_I, (float4*)w.S);
    ++*nl;
    return cudaGetLastError();
}

cudaError_t cd_launch_pack(const CdGeom& g, const CdWork& w, const double* vel, const double* omega,
                           const double* radius, const double* inv_m, const double* inv_I, const double* f_ext,
                           int free_flight, int precision, cudaStream_t s, int* nl)
{
    (void)radius; (void)inv_I;
    int gb = grid_n(g.n);
    if (g.dim == 2) {
        if (precision == CD_FP64) k_pack<2, double><<<gb, CD_BLOCK, 0, s>>>(g, w, vel, omega, inv_m, f_ext, free_flight);
        else k_pack<2, float><<<gb, CD_BLOCK, 0, s>>>(g, w, vel, omega, inv_m, f_ext, free_flight);
        ++*nl;
    } else {
        if (precision == CD_FP64) k_pack<3, double><<<gb, CD_BLOCK, 0, s>>>(g, w, vel, omega, inv_m, f_ext, free_flight);
        else k_pack<3, float><<<gb, CD_BLOCK, 0, s>>>(g, w, vel, omega, inv_m, f_ext, free_flight);
        ++*nl;
    }
    return cudaGetLastError();
}

cudaError_t cd_launch_unpack(const CdGeom& g, const CdWork& w, double* pos, double* vel, double* omega,
                             double* theta, int integrate, int precision, cudaStream_t s, int* nl)
{
    int gb = grid_n(g.n);
    if (g.dim == 2) {
        if (precision == CD_FP64) k_unpack<2, double><<<gb, CD_BLOCK, 0, s>>>(g, w, pos, vel, omega, theta, integrate);
        else k_unpack<2, float><<<gb, CD_BLOCK, 0, s>>>(g, w, pos, vel, omega, theta, integrate);
        ++*nl;
    } else {
        if (precision == CD_FP64) k_unpack<3, double><<<gb, CD_BLOCK, 0, s>>>(g, w, pos, vel, omega, theta, integrate);
        else k_unpack<3, float><<<gb, CD_BLOCK, 0, s>>>(g, w, pos, vel, omega, theta, integrate);
        ++*nl;
    }
    return cudaGetLastError();
}

// Kernel of each schedule: 0 colour barrier, 3 batched, 4 mixed update,
// 5 domain-wise update, 6 merged last colours.
static int sweep_kind(const CdGeom& g)
{
    if (g.npk > 1) return 3;
    if (g.par_p > 0.0) return 4;
    if (g.ndom_total > 1) return 5;
    if (g.merge_last) return 6;
    return 0;
}

static const void* sweep_fn(int dim, int precision, int kind)
{
    if (kind == 6) {
        if (dim == 2)
            return precision == CD_FP64 ? (const void*)k_sweep<2, double, CD_SWEEP_MERGE>
                                        : (const void*)k_sweep<2, float, CD_SWEEP_MERGE>;
        return precision == CD_FP64 ? (const void*)k_sweep<3, double, CD_SWEEP_MERGE>
                                    : (const void*)k_sweep<3, float, CD_SWEEP_MERGE>;
    }
    if (kind == 5) {
        if (dim == 2)
            return precision == CD_FP64 ? (const void*)k_sweep<2, double, CD_SWEEP_DOMAINS>
                                        : (const void*)k_sweep<2, float, CD_SWEEP_DOMAINS>;
        return precision == CD_FP64 ? (const void*)k_sweep<3, double, CD_SWEEP_DOMAINS>
                                    : (const void*)k_sweep<3, float, CD_SWEEP_DOMAINS>;
    }
    if (kind == 4) {
        if (dim == 2)
            return precision == CD_FP64 ? (const void*)k_sweep<2, double, CD_SWEEP_MIXED>
                                        : (const void*)k_sweep<2, float, CD_SWEEP_MIXED>;
        return precision == CD_FP64 ? (const void*)k_sweep<3, double, CD_SWEEP_MIXED>
                                    : (const void*)k_sweep<3, float, CD_SWEEP_MIXED>;
    }
    if (kind == 3) {
        if (dim == 2)
            return precision == CD_FP64 ? (const void*)k_sweep_batch<2, double> : (const void*)k_sweep_batch<2, float>;
        return precision == CD_FP64 ? (const void*)k_sweep_batch<3, double> : (const void*)k_sweep_batch<3, float>;
    }
    if (dim == 2)
        return precision == CD_FP64 ? (const void*)k_sweep<2, double, CD_SWEEP_PLAIN>
                                    : (const void*)k_sweep<2, float, CD_SWEEP_PLAIN>;
    return precision == CD_FP64 ? (const void*)k_sweep<3, double, CD_SWEEP_PLAIN>
                                : (const void*)k_sweep<3, float, CD_SWEEP_PLAIN>;
}

static const int kSweepKinds[] = {0, 3, 4, 5, 6};

// Blocks of the cooperative sweep grid: one per SM (keeps the grid barrier
// cheap), for whichever of the kernels the system uses.
int cd_sweep_max_blocks(int precision, int dim, int num_sms)
{
    for (int kind : kSweepKinds) {
        int b = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, sweep_fn(dim, precision, kind), CD_SWEEP_THREADS, 0) !=
            cudaSuccess)
            return 0;
        if (b < 1) return 0;
    }
    return num_sms;
}

// 1 if `per_sm` blocks of `threads` threads of the sweep kernel the system
// uses can be resident on one SM.
int cd_sweep_fits(const CdGeom& g, int precision, int threads, int per_sm)
{
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, sweep_fn(g.dim, precision, sweep_kind(g)), threads, 0) !=
        cudaSuccess)
        return 0;
    return b >= per_sm ? 1 : 0;
}

cudaError_t cd_launch_sweep(const CdGeom& g, const CdWork& w, int coop_blocks, int threads, int precision,
                            int criterion, double alpha, int max_sweeps, int pw, cudaStream_t s, int* nl)
{
    (void)pw;
    cudaError_t e = cudaMemsetAsync(w.ctrl, 0, 2 * sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    CdGeom ga = g;
    CdWork wa = w;
    int crit = criterion;
    double al = alpha;
    int ms = max_sweeps;
    void* args[] = {&ga, &wa, &crit, &al, &ms};
    const int kind = sweep_kind(g);
    ++*nl;
    return cudaLaunchCooperativeKernel(sweep_fn(g.dim, precision, kind), dim3(coop_blocks), dim3(threads),
                                       args, 0, s);
}
