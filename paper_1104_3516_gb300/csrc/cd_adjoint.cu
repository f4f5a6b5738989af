// cd_adjoint.cu -- reverse-mode derivative of one CD time step (2D, FP64)
// at fixed contact states, and the tape the forward steps record for it.
//
// The paper differentiates nothing; the derivative is that of the step map
// (x, v, omega, mu) -> (x', v', omega') of Eqs. 1-2 with the converged
// impulses of the iteration (Sec. 2.1, Fig. 2, Eqs. 3-11).  Once converged,
// every contact is open (P = 0, Eq. 3), sticking (Eq. 5: the gap closes,
// u_n' = -g/dt, and there is no slip, u_t' = 0) or sliding (Eqs. 9-11:
// u_n' = -g/dt and P_t = s mu P_n).  With the states frozen these are linear
// in the impulses: S (H v' + g/dt) = 0 with v' = v_free + W H^T Phi p, where
// H maps body velocities to contact-frame relative velocities, W = diag(1/m,
// 1/m, 1/I), S keeps the rows above and Phi maps the free impulse components
// p to (P_n, P_t).  The reverse pass for an incoming gradient lambda of v'
// (plus dt times that of x', Eq. 2) solves the transposed system
//     Phi^T H Gamma = 0,   Gamma = W (lambda - H^T Y)
// for the multipliers Y by Gauss-Seidel in the same colour order as the
// forward sweep: per contact u = H Gamma, then Y += M (u_n, u_t) for a
// sticking contact, Y_n += m_n (u_n + s mu u_t) for a sliding one, and Gamma
// -= W H^T dY on the two bodies.  Then
//     dL/dv_free = lambda - H^T Y        (= dL/dv, dL/domega of the step's input)
//     dL/dmu     = sum_sliding s P_n (H Gamma)_t
//     dL/dx      = dL/dx' + sum over contacts of the derivative through the
//                  normal n and the gap g:  dL/dn = P_n dGamma + P_t R^T dGamma
//                  - Y_n dv' - Y_t R^T dv',  dL/dg = -Y_n / dt,
//                  with dGamma, dv' the differences body b - body a and
//                  R^T (u_x, u_y) = (u_y, -u_x); for a pair dn/dd = (I - n n^T)
//                  / |d|, dg/dd = n, d = x_b - x_a; for a wall dg/dx_a = -n.
// A loss that also depends on the step's wall forces (sum of the normal
// impulses on wall k over dt) adds q_n = dL/dF_k / dt to u_n on that wall's
// contacts: the rows solved become Phi^T (H Gamma + q) = 0.
// With params.adjoint_compliance eps > 0 each retained row is softened to
// Phi^T (H Gamma + q) - eps diag(w_n, w_t) Y = 0 (contacts with a small
// compliance), which makes the transposed system nonsingular on hyperstatic
// networks, where the rigid one has no unique multipliers.
// A contact whose normal impulse is at most CD_GRAZING times the step's
// largest is taken as open (two bodies left touching by an inelastic
// collision carry rounding noise there, and the map has a kink).
#include "cd_flow_core.cuh"

namespace {

__device__ __forceinline__ double warp_sum_a(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ double warp_max_a(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Block sum of NV values per thread (fixed tree); valid in thread 0.
template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV], double (*s_red)[4])
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int j = 0; j < NV; ++j) v[j] = warp_sum_a(v[j]);
    if (lane == 0)
#pragma unroll
        for (int j = 0; j < NV; ++j) s_red[wid][j] = v[j];
    __syncthreads();
    if (wid == 0) {
        const int nw = blockDim.x >> 5;
#pragma unroll
        for (int j = 0; j < NV; ++j) v[j] = warp_sum_a(lane < nw ? s_red[lane][j] : 0.0);
    }
    __syncthreads();
}

// Sum (or max) over the blocks' partials, identical in every block.
template <bool MAX>
__device__ __forceinline__ double grid_reduce(const double* part, int nb, double* s_bc)
{
    if (threadIdx.x < 32) {
        double x = 0.0;
        for (int b = threadIdx.x; b < nb; b += 32) x = MAX ? fmax(x, part[b]) : x + part[b];
        x = MAX ? warp_max_a(x) : warp_sum_a(x);
        if (threadIdx.x == 0) *s_bc = x;
    }
    __syncthreads();
    const double r = *s_bc;
    __syncthreads();
    return r;
}

__device__ __forceinline__ bool is_slide(double mu, const double2& P)
{
    return fabs(P.y) == mu * P.x;
}

#define ADJ_WARPS 12
#define ADJ_THREADS (32 * ADJ_WARPS)
#define ADJ_REC 12   // 64-bit elements of a particle: Gamma, Lambda, the position gradient, 4 each
#define ADJ_OPEN 0xffffffffu   // adj_ord of an open contact

// What the block's warps share.
struct AdjShared {
    int off[CD_KMAX + 1];
    int lo[CD_KMAX], end[CD_KMAX];     // this block's positions of each colour
    int base[CD_KMAX + 1];             // first of its warp items (32 contacts)
    double acc[2][ADJ_WARPS][32];      // |Y| and |dY| of a sweep by lane
    double sum[2];
    int dead;                          // a wait gave up
    int state;                         // 0: another sweep; 1: converged; 2: diverged
    double resid;
};

__device__ __forceinline__ u64* adj_gamma(const CdWork& w, int i) { return w.adj_rec + (size_t)ADJ_REC * i; }
__device__ __forceinline__ u64* adj_lambda(const CdWork& w, int i) { return w.adj_rec + (size_t)ADJ_REC * i + 4; }
__device__ __forceinline__ u64* adj_gx(const CdWork& w, int i) { return w.adj_rec + (size_t)ADJ_REC * i + 8; }

// a x + c y, the first product fused: sums of two products are written out, since
// gradients lose seven digits to cancellation (pyramids: 4e-13 of 1.5e-4) and
// another order gives other last digits.
__device__ __forceinline__ double two(double a, double x, double c, double y)
{
    return __fma_rn(a, x, __dmul_rn(c, y));
}

// |(x, y)| for the sweep's sums.  The square root (the forward solve's integer
// form is up to 7.3e-15 off, which the residual would carry); its overflow and NaN
// tell the test that the iteration diverged.
__device__ __forceinline__ double adj_abs(double x, double y)
{
    return sqrt(x * x + y * y);
}

// A non-open contact's data that no sweep changes.
struct AdjContact {
    int2 ab;
    bool wall, slide;
    double nx, ny, mn, mt, s;   // s: direction of sliding
    double4_16a sa, sb;
};

__device__ __forceinline__ AdjContact adj_load(const CdGeom& g, const CdWork& w, const CdTape& t, int p)
{
    AdjContact c;
    const double2 P = t.P[p];
    c.ab = t.ab[p];
    c.wall = c.ab.y >= g.n;
    const double4_16a geo = t.geo[p];
    c.nx = geo.x; c.ny = geo.y; c.mn = geo.w; c.mt = t.mt[p];
    const double4_16a* S = (const double4_16a*)w.S;
    c.sa = S[c.ab.x];
    c.sb = c.wall ? make_double4_16a(0.0, 0.0, 0.0, 0.0) : S[c.ab.y];
    c.slide = is_slide(g.mu, P);
    c.s = (P.y < 0.0) ? -1.0 : 1.0;
    return c;
}

// One Gauss-Seidel update of the transposed system on a contact: Ga, Gb and Y
// change, dY is the step.
__device__ __forceinline__ void adj_update(const CdGeom& g, const CdAdjIO& io, const AdjContact& c, double inv1e,
                                           Vec<double>::V4& Ga, Vec<double>::V4& Gb, double2& Y, double2& dY,
                                           double2& f)
{
    const double dgx = Gb.x - Ga.x, dgy = Gb.y - Ga.y;
    const double un = two(dgx, c.nx, dgy, c.ny) + (c.wall ? io.wq[c.ab.y - g.n] : 0.0);
    const double ut = two(dgy, c.nx, -dgx, c.ny) - two(c.sa.y, Ga.z, c.sb.y, Gb.z);
    // with compliance eps the rows are Phi^T (H Gamma + q) - eps diag(w) Y = 0
    const double eps = io.eps;
    if (c.slide) {
        dY.x = c.mn * (un + c.s * g.mu * ut);
        dY.y = 0.0;
    } else {
        dY.x = c.mn * un;
        dY.y = c.mt * ut;
    }
    if (eps != 0.0) {
        dY.x = (dY.x - eps * Y.x) * inv1e;
        if (!c.slide) dY.y = (dY.y - eps * Y.y) * inv1e;
    }
    f.x = two(dY.x, c.nx, -dY.y, c.ny);
    f.y = two(dY.x, c.ny, dY.y, c.nx);
    // Gamma -= W H^T dY (body a: -f, -r_a dY_t; body b: +f, -r_b dY_t)
    Ga.x += c.sa.x * f.x; Ga.y += c.sa.x * f.y; Ga.z += c.sa.z * dY.y;
    if (!c.wall) {
        Gb.x -= c.sb.x * f.x; Gb.y -= c.sb.x * f.y; Gb.z += c.sb.z * dY.y;
    }
    Y.x += dY.x;
    Y.y += dY.y;
}

// The contact's part of dL/dmu, and of the position gradient through its
// normal and gap: dL/dg, and for a pair what body a loses and b gains.
__device__ __forceinline__ double adj_geometry(const CdGeom& g, const CdTape& t, const AdjContact& c, int p,
                                               const Vec<double>::V4& Ga, const Vec<double>::V4& Gb, double2 Y,
                                               double& dLg, double2& dd)
{
    const double2 P = t.P[p];
    const double4_16a va = t.V[c.ab.x];
    double4_16a vb = make_double4_16a(0.0, 0.0, 0.0, 0.0);
    if (!c.wall) vb = t.V[c.ab.y];
    else {
        const double* u = g.wall_vel + 3 * (c.ab.y - g.n);
        vb.x = u[0];
        vb.y = u[1];
    }
    const double dgx = Gb.x - Ga.x, dgy = Gb.y - Ga.y;
    const double dvx = vb.x - va.x, dvy = vb.y - va.y;
    double dmu = 0.0;
    if (c.slide) dmu = c.s * P.x * (two(dgy, c.nx, -dgx, c.ny) - two(c.sa.y, Ga.z, c.sb.y, Gb.z));
    dLg = -Y.x / g.dt;
    dd = make_double2(0.0, 0.0);
    if (c.wall) return dmu;
    const double dLnx = two(P.x, dgx, P.y, dgy) - Y.x * dvx - Y.y * dvy;
    const double dLny = two(P.x, dgy, -P.y, dgx) - Y.x * dvy + Y.y * dvx;
    const double dist = t.geo[p].z * g.dt + c.sa.y + c.sb.y;   // |d| = g + r_a + r_b
    const double nd = two(c.nx, dLnx, c.ny, dLny);
    dd.x = (dLnx - c.nx * nd) / dist + dLg * c.nx;
    dd.y = (dLny - c.ny * nd) / dist + dLg * c.ny;
    return dmu;
}

// Records the step in the tape's next slot (of T); the last block to have read
// the slot advances it.
__global__ void k_tape_record(CdWork w, int n, int64_t cap, int T)
{
    CdCtrl* ctrl = w.ctrl;
    const int slot = ctrl->tape_slot;
    const CdTape t = cd_tape_slot(w.tape, n, cap, slot);
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(&ctrl->tape_ticket, 1) == (int)gridDim.x - 1) {
        ctrl->tape_ticket = 0;
        ctrl->tape_slot = (slot + 1) % T;
    }
    const int nc = ctrl->nc;
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int stride = gridDim.x * blockDim.x;
    if (tid == 0) {
        t.hdr->nc = nc;
        t.hdr->ncolours = ctrl->ncolours;
        t.hdr->valid = (ctrl->skip == 0 && ctrl->error == CDE_NONE) ? 1 : 0;
    }
    for (int k = tid; k <= CD_KMAX; k += stride) t.hdr->colour_off[k] = w.colour_off[k];
    for (int c = tid; c < nc; c += stride) {
        t.ab[c] = w.c_ab[c];
        t.geo[c] = ((const double4_16a*)w.c_geo)[c];
        t.mt[c] = ((const double*)w.c_m)[c];
        t.P[c] = ((const double2*)w.c_P)[c];
    }
    for (int i = tid; i < n; i += stride) t.V[i] = ((const double4_16a*)w.V)[i];
}

__global__ void k_set_tape_slot(CdCtrl* ctrl, int slot)
{
    ctrl->tape_slot = slot;
}

// The block's sum of x (lane sums in sh.acc[q]), left for the other blocks and
// gathered from them: one warp.  Every block adds the same sums in the same order.
__device__ __forceinline__ bool adj_gather(CdCtrl* ctrl, AdjShared& sh, FlowSum* row, int q, unsigned tag)
{
    const int lane = threadIdx.x & 31, nb = gridDim.x;
    double v[ADJ_WARPS];
#pragma unroll
    for (int u = 0; u < ADJ_WARPS; ++u) v[u] = sh.acc[q][u][lane];
    double x = flow_sum_warp(v);
    if (lane == 0) flow_sum_store(row + blockIdx.x, x, tag);
    FlowBound bound;
    for (int b0 = 0; b0 < nb; b0 += 160) {
        u64 f[5][2];
        double y[5];
        bool have = false;
        while (!__all_sync(0xffffffffu, have)) {
            have = true;
#pragma unroll
            for (int u = 0; u < 5; ++u)
                if (b0 + 32 * u + lane < nb) flow_load(row[b0 + 32 * u + lane].e, f[u]);
#pragma unroll
            for (int u = 0; u < 5; ++u) {
                const bool in = b0 + 32 * u + lane < nb;
                have = have && (!in || flow_sum_is(f[u], tag));
                y[u] = in ? flow_sum_of(f[u]) : 0.0;
            }
            if (!__all_sync(0xffffffffu, bound.go(ctrl))) {
                *(volatile int*)&sh.dead = 1;
                return false;
            }
        }
        const double z = flow_sum_warp(y);
        x = b0 ? x + z : z;
    }
    if (lane == 0) sh.sum[q] = x;
    return true;
}

// The whole reverse step as one cooperative kernel: initial Gamma, the
// Gauss-Seidel sweeps of the transposed system, the position gradient, the
// outputs.  The sweeps and the gradient run by dataflow as the forward solve
// does (cd_flow.cu): a particle's Gamma carries the number of its updates, and a
// contact waits for its two records, not for a colour.  Only contacts that are
// not open take part (of a settling packing's, one in a hundred).  A sweep's
// sums of |Y| and |dY| end it: two warps gather them from all blocks.  What bounds it: the update's ~25
// dependent FP64 instructions of 64 cycles, the way of a record between SMs
// (~850 cycles) and, once a sweep, that of the sums and the test.  3,334 sliding
// pyramids, 48 sweeps of two colours: 714 us with a grid barrier a colour, 486
// now; 10,000 settling discs, one or two sweeps: 53 -> 38 us.
__global__ void __launch_bounds__(ADJ_THREADS, 1)
k_adjoint(CdGeom g, CdWork w, CdTape t, CdAdjIO io, double alpha, int max_sweeps)
{
    typedef FlowBody<2, double> Record;
    typedef Vec<double>::V4 V4;
    __shared__ AdjShared sh;
    __shared__ double s_red[ADJ_WARPS][4];
    __shared__ double s_bc;
    CdCtrl* ctrl = w.ctrl;
    const int nb = gridDim.x;
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int stride = gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (!t.hdr->valid) {
        if (tid == 0) atomicCAS(&ctrl->error, CDE_NONE, CDE_TAPE);
        return;
    }
    const int n = g.n;
    const int nc = t.hdr->nc;
    const int K = t.hdr->ncolours;
    FlowSum* part = (FlowSum*)w.adj_part;   // rows: |Y| and |dY| of even, then of odd sweeps
    unsigned long long epoch = 0;
    // this block's positions of each colour: whole warp items, their remainders from another block on each
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        const int lo = t.hdr->colour_off[k], hi = t.hdr->colour_off[k + 1];
        const long long items = (hi - lo + 31) >> 5;
        const int r = (int)(((long long)k * 5 * nb >> 3) % nb);
        const int i0 = (int)((items * blockIdx.x + r) / nb), i1 = (int)((items * (blockIdx.x + 1) + r) / nb);
        sh.lo[k] = min(lo + (i0 << 5), hi);
        sh.end[k] = min(lo + (i1 << 5), hi);
        sh.base[k + 1] = i1 - i0;
    }
    if (threadIdx.x == 0) { sh.dead = 0; sh.state = (nc == 0) ? 1 : 0; sh.resid = 0.0; }
    if (threadIdx.x < 4) flow_sum_store(part + (size_t)threadIdx.x * nb + blockIdx.x, 0.0, 0u);

    // incoming gradient: lambda = dL/dv' + dt dL/dx' (Eq. 2), Gamma = W lambda
    const double4_16a* S = (const double4_16a*)w.S;
    for (int i = tid; i < n; i += stride) {
        const double lx = io.dLv[2 * i] + g.dt * io.dLx[2 * i];
        const double ly = io.dLv[2 * i + 1] + g.dt * io.dLx[2 * i + 1];
        const double lw = io.dLw[i];
        const double im = S[i].x;
        const double iI = g.rotations ? io.inv_I[i] : 0.0;
        V4 v;
        v.x = im * lx; v.y = im * ly; v.z = iI * lw; v.w = 0.0;
        Record G;
        G.pack(v, v, 0u);
        G.store(adj_gamma(w, i));
        v.x = v.y = v.z = 0.0;
        G.pack(v, v, 0u);
        G.store(adj_lambda(w, i));
        v.x = io.dLx[2 * i]; v.y = io.dLx[2 * i + 1];
        G.pack(v, v, 0u);
        G.store(adj_gx(w, i));
        w.adj_lam[i] = make_double4_16a(lx, ly, lw, 0.0);
        w.adj_mask[i] = 0ULL;
    }
    {
        double pmax = 0.0;
        for (int c = tid; c < nc; c += stride) pmax = fmax(pmax, t.P[c].x);
        pmax = warp_max_a(pmax);
        if (lane == 0) s_red[wid][0] = pmax;
        __syncthreads();
        if (threadIdx.x == 0) {
            double m = 0.0;
            for (int q = 0; q < ADJ_WARPS; ++q) m = fmax(m, s_red[q][0]);
            w.partials[blockIdx.x] = m;
            sh.base[0] = 0;
            for (int k = 0; k < K; ++k) sh.base[k + 1] += sh.base[k];
        }
    }
    if (!cd_grid_sync(ctrl, nb, epoch)) return;
    // the open threshold, from the largest normal impulse; the colours of each
    // particle's contacts; and the scale of the multipliers that the incoming
    // gradient calls for, sum of m_n (|Gamma_a| + |Gamma_b|)
    const double thr = CD_GRAZING * grid_reduce<true>(w.partials, nb, &s_bc);
    for (int k = 0; k < K; ++k)
        for (int p = sh.lo[k] + (int)threadIdx.x; p < sh.end[k]; p += blockDim.x) {
            if (!(t.P[p].x > thr)) continue;
            const int2 ab = t.ab[p];
            atomicOr(&w.adj_mask[ab.x], 1ULL << k);
            if (ab.y < n) atomicOr(&w.adj_mask[ab.y], 1ULL << k);
        }
    {
        double acc[1] = {0.0};
        for (int c = tid; c < nc; c += stride) {
            const int2 ab = t.ab[c];
            Record G;
            V4 Ga, Gb, o;
            G.load(adj_gamma(w, ab.x));
            G.unpack(Ga, o);
            double sc = sqrt(Ga.x * Ga.x + Ga.y * Ga.y) + S[ab.x].y * fabs(Ga.z);
            if (ab.y < n) {
                G.load(adj_gamma(w, ab.y));
                G.unpack(Gb, o);
                sc += sqrt(Gb.x * Gb.x + Gb.y * Gb.y) + S[ab.y].y * fabs(Gb.z);
            } else {
                sc += fabs(io.wq[ab.y - n]);
            }
            acc[0] += t.geo[c].w * sc;
        }
        block_sum<1>(acc, s_red);
        if (threadIdx.x == 0) w.partials[nb + blockIdx.x] = acc[0];
    }
    if (!cd_grid_sync(ctrl, nb, epoch)) return;
    const double yscale = grid_reduce<false>(w.partials + nb, nb, &s_bc);
    // a contact's place among each particle's contacts and their number (8 bits each)
    double nstick = 0.0, nslide = 0.0, nmark = 0.0;
    for (int k = 0; k < K; ++k)
        for (int p = sh.lo[k] + (int)threadIdx.x; p < sh.end[k]; p += blockDim.x) {
            unsigned ord = ADJ_OPEN;
            const double2 P = t.P[p];
            if (P.x > thr) {
                const int2 ab = t.ab[p];
                const u64 below = (1ULL << k) - 1ULL;
                const u64 ma = w.adj_mask[ab.x], mb = (ab.y < n) ? w.adj_mask[ab.y] : 0ULL;
                ord = (unsigned)__popcll(ma & below) | ((unsigned)__popcll(ma) << 8) |
                      ((unsigned)__popcll(mb & below) << 16) | ((unsigned)__popcll(mb) << 24);
                w.adj_Y[p] = make_double2(0.0, 0.0);
                if (is_slide(g.mu, P)) nslide += 1.0;
                else nstick += 1.0;
            }
            w.adj_ord[p] = ord;
        }
    for (int i = tid; i < n; i += stride) nmark += w.adj_mask[i] != 0ULL ? 1.0 : 0.0;
    __syncthreads();

    // sweeps until sum |dY| <= alpha max(sum |Y|, yscale)
    const int Q = sh.base[K];
    const bool single = Q <= ADJ_WARPS;   // a warp's one item stays in its registers
    const double inv1e = 1.0 / (1.0 + io.eps), most = 1e30 * fmax(yscale, 1e-300);
    int sweeps = 0;
    AdjContact c;
    double2 Y = make_double2(0.0, 0.0);
    unsigned ord = ADJ_OPEN;
    while (sh.state == 0 && sweeps < max_sweeps) {
        double ay = 0.0, ad = 0.0;
        int k = 0;
        for (int q = wid; q < Q; q += ADJ_WARPS) {
            while (q >= sh.base[k + 1]) ++k;
            const int p = sh.lo[k] + 32 * (q - sh.base[k]) + lane;
            if (!single || sweeps == 0) {
                ord = (p < sh.end[k]) ? w.adj_ord[p] : ADJ_OPEN;
                if (ord != ADJ_OPEN) {
                    c = adj_load(g, w, t, p);
                    Y = w.adj_Y[p];
                }
            }
            const bool act = ord != ADJ_OPEN;
            if (!__any_sync(0xffffffffu, act)) continue;
            Record A, B;
            const unsigned ta = (unsigned)sweeps * ((ord >> 8) & 255u) + (ord & 255u);
            const unsigned tb = (unsigned)sweeps * (ord >> 24) + ((ord >> 16) & 255u);
            u64* pa = act ? adj_gamma(w, c.ab.x) : nullptr;
            u64* pb = (act && !c.wall) ? adj_gamma(w, c.ab.y) : nullptr;
            if (!flow_wait<2, double>(ctrl, &sh.dead, pa, ta, pb, tb, A, B, !pa, !pb)) break;
            double2 dY = make_double2(0.0, 0.0), f = dY;
            V4 Ga, Gb, o;
            if (act) {
                A.unpack(Ga, o);
                Gb.x = Gb.y = Gb.z = Gb.w = 0.0;
                if (pb) B.unpack(Gb, o);
                adj_update(g, io, c, inv1e, Ga, Gb, Y, dY, f);
                A.pack(Ga, Ga, ta + 1u);
                A.store(pa);
                if (pb) {
                    B.pack(Gb, Gb, tb + 1u);
                    B.store(pb);
                }
                w.adj_Y[p] = Y;
                ay += adj_abs(Y.x, Y.y);
                ad += adj_abs(dY.x, dY.y);
            }
            // Lambda follows in its own record, which nobody else waits for now
            pa = act ? adj_lambda(w, c.ab.x) : nullptr;
            pb = (act && !c.wall) ? adj_lambda(w, c.ab.y) : nullptr;
            if (!flow_wait<2, double>(ctrl, &sh.dead, pa, ta, pb, tb, A, B, !pa, !pb)) break;
            if (act) {
                V4 L;
                A.unpack(L, o);
                L.x -= f.x; L.y -= f.y; L.z -= c.sa.y * dY.y;
                A.pack(L, L, ta + 1u);
                A.store(pa);
                if (pb) {
                    B.unpack(L, o);
                    L.x += f.x; L.y += f.y; L.z -= c.sb.y * dY.y;
                    B.pack(L, L, tb + 1u);
                    B.store(pb);
                }
            }
        }
        sh.acc[0][wid][lane] = ay;
        sh.acc[1][wid][lane] = ad;
        __syncthreads();
        if (sh.dead) return;
        if (wid < 2) adj_gather(ctrl, sh, part + (size_t)(2 * (sweeps & 1) + wid) * nb, wid, (unsigned)sweeps + 1u);
        __syncthreads();
        if (sh.dead) return;
        ++sweeps;
        if (threadIdx.x == 0) {
            const double ysum = sh.sum[0], dsum = sh.sum[1];
            const double den = fmax(ysum, yscale);
            if (dsum <= alpha * den) sh.state = 1;
            if (!(ysum <= most)) sh.state = 2;   // growing without bound, or not finite
            if (sh.state || sweeps == max_sweeps) sh.resid = (den > 0.0) ? dsum / den : 0.0;
        }
        __syncthreads();
    }

    // position gradient, each particle's contacts in the order of their colours
    double dmu = 0.0;
    if (sweeps > 0) {
        int k = 0;
        for (int q = wid; q < Q; q += ADJ_WARPS) {
            while (q >= sh.base[k + 1]) ++k;
            const int p = sh.lo[k] + 32 * (q - sh.base[k]) + lane;
            if (!single) {
                ord = (p < sh.end[k]) ? w.adj_ord[p] : ADJ_OPEN;
                if (ord != ADJ_OPEN) {
                    c = adj_load(g, w, t, p);
                    Y = w.adj_Y[p];
                }
            }
            const bool act = ord != ADJ_OPEN;
            if (!__any_sync(0xffffffffu, act)) continue;
            Record A, B;
            V4 v, o;
            double dLg = 0.0;
            double2 dd = make_double2(0.0, 0.0);
            u64* pa = act ? adj_gamma(w, c.ab.x) : nullptr;
            u64* pb = (act && !c.wall) ? adj_gamma(w, c.ab.y) : nullptr;
            // (every block's sweeps are known to be done; the records say so themselves)
            if (!flow_wait<2, double>(ctrl, &sh.dead, pa, (unsigned)sweeps * ((ord >> 8) & 255u), pb,
                                      (unsigned)sweeps * (ord >> 24), A, B, !pa, !pb)) break;
            if (act) {
                V4 Gb;
                A.unpack(v, o);
                Gb.x = Gb.y = Gb.z = Gb.w = 0.0;
                if (pb) B.unpack(Gb, o);
                dmu += adj_geometry(g, t, c, p, v, Gb, Y, dLg, dd);
                pa = adj_gx(w, c.ab.x);
                if (pb) pb = adj_gx(w, c.ab.y);
            }
            if (!flow_wait<2, double>(ctrl, &sh.dead, pa, ord & 255u, pb, (ord >> 16) & 255u, A, B, !pa, !pb)) break;
            if (act) {
                A.unpack(v, o);
                if (c.wall) {
                    v.x -= dLg * c.nx; v.y -= dLg * c.ny;
                } else {
                    v.x -= dd.x; v.y -= dd.y;
                }
                A.pack(v, v, (ord & 255u) + 1u);
                A.store(pa);
                if (pb) {
                    B.unpack(v, o);
                    v.x += dd.x; v.y += dd.y;
                    B.pack(v, v, ((ord >> 16) & 255u) + 1u);
                    B.store(pb);
                }
            }
        }
    }
    double acc4[4] = {dmu, nstick, nslide, nmark};
    __syncthreads();
    if (sh.dead) return;
    block_sum<4>(acc4, s_red);
    if (threadIdx.x == 0)
        for (int q = 0; q < 4; ++q) w.partials[q * nb + blockIdx.x] = acc4[q];
    if (!cd_grid_sync(ctrl, nb, epoch)) return;
    for (int i = tid; i < n; i += stride) {
        const double4_16a lam = w.adj_lam[i];
        Record X;
        V4 v, o;
        X.load(adj_gx(w, i));
        X.unpack(v, o);
        io.ox[2 * i] = v.x;
        io.ox[2 * i + 1] = v.y;
        X.load(adj_lambda(w, i));
        X.unpack(v, o);
        io.ov[2 * i] = lam.x - v.x;
        io.ov[2 * i + 1] = lam.y - v.y;
        io.ow[i] = lam.z - v.z;
    }
    if (blockIdx.x == 0) {
        double r[4];
        for (int q = 0; q < 4; ++q) r[q] = grid_reduce<false>(w.partials + q * nb, nb, &s_bc);
        if (threadIdx.x == 0) {
            ctrl->adj_sweeps = sweeps;
            ctrl->adj_converged = sh.state == 1;
            ctrl->adj_residual = sh.resid;
            ctrl->adj_dmu = r[0];
            ctrl->adj_nc = nc;
            ctrl->adj_nstick = (long long)r[1];
            ctrl->adj_nslide = (long long)r[2];
            ctrl->adj_nbodies = (long long)r[3];
            ctrl->adj_diverged = sh.state == 2;
            ctrl->tape_slot = io.slot;   // the step is consumed
        }
    }
}

}  // namespace

cudaError_t cd_launch_tape_record(const CdGeom& g, const CdWork& w, int64_t cap, int T, cudaStream_t s, int* nl)
{
    int blocks = (g.n + CD_BLOCK - 1) / CD_BLOCK;
    if (blocks < 64) blocks = 64;
    if (blocks > 4096) blocks = 4096;
    k_tape_record<<<blocks, CD_BLOCK, 0, s>>>(w, g.n, cap, T);
    ++*nl;
    return cudaGetLastError();
}

cudaError_t cd_launch_set_tape_slot(const CdWork& w, int slot, cudaStream_t s, int* nl)
{
    k_set_tape_slot<<<1, 1, 0, s>>>(w.ctrl, slot);
    ++*nl;
    return cudaGetLastError();
}

int cd_adjoint_blocks_per_sm()
{
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_adjoint, ADJ_THREADS, 0) != cudaSuccess) return 0;
    return b;
}

cudaError_t cd_launch_adjoint(const CdGeom& g, const CdWork& w, const CdTape& t, const CdAdjIO& io, double alpha,
                              int max_sweeps, int coop_blocks, cudaStream_t s, int* nl)
{
    cudaError_t e = cudaMemsetAsync(w.ctrl, 0, 2 * sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    CdGeom ga = g;
    CdWork wa = w;
    CdTape ta = t;
    CdAdjIO ia = io;
    double al = alpha;
    int ms = max_sweeps;
    void* args[] = {&ga, &wa, &ta, &ia, &al, &ms};
    ++*nl;
    return cudaLaunchCooperativeKernel((const void*)k_adjoint, dim3(coop_blocks), dim3(ADJ_THREADS), args, 0, s);
}
