// cd_detect_core.cuh -- the pieces of contact detection (paper Sec. 3.2) and of
// the contact geometry (Sec. 2.1) that the detection kernels share.
#pragma once

#include <climits>

#include "cd_internal.cuh"

// ---------------------------------------------------------------------------
// Cell list.  Every packing of a batched system has its own grid (a plain
// system is one packing); global cell id = the packing's cell_base + local id,
// so particles of different packings are never in neighbouring cells.
// ---------------------------------------------------------------------------
// Candidates a lane looks at together.  The walk is a chain of two dependent
// loads a candidate (id, then position): four chains at once take the counting
// pass of a million spheres from 335 to 231 us (two: 5 us more).
#define CD_WALK 4
#define CD_QUEUE (32 * (CD_WALK + 1))   // queued pairs of a warp

struct GridV {
    double lo[3], cs[3], inv_cs[3], L[3];
    int ncell[3], periodic[3];
    int base, wall_mask, pkid;
};

__device__ __forceinline__ void grid_of(const CdGeom& g, const CdWork& w, int i, GridV& v)
{
    if (g.npk > 1) {
        const int b = w.pack_of[i];
        const CdPack& p = w.pk[b];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            v.lo[k] = p.lo[k]; v.cs[k] = p.cs[k]; v.inv_cs[k] = p.inv_cs[k]; v.L[k] = p.L[k];
            v.ncell[k] = p.ncell[k]; v.periodic[k] = p.periodic[k];
        }
        v.base = p.cell_base; v.wall_mask = p.wall_mask; v.pkid = b;
    } else {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            v.lo[k] = g.lo[k]; v.cs[k] = g.cs[k]; v.inv_cs[k] = g.inv_cs[k]; v.L[k] = g.L[k];
            v.ncell[k] = g.ncell[k]; v.periodic[k] = g.periodic[k];
        }
        v.base = 0; v.wall_mask = g.wall_mask; v.pkid = 0;
    }
}

// Cell index along axis k: floor((x - lo) / cs) clamped to the grid, with
// the quotient taken as a product by 1 / cs and rounded down to an integer
// in one conversion (a correctly rounded FP64 division is ~10 FP64
// instructions).  Either rounding may put a particle within a few ulps of a
// cell face into the neighbouring cell; no contact is lost: a contact is
// closer than r_a + r_b + delta <= 2 r_max + delta, the cell side is longer
// than that by a relative 1e-9 (far more than the misplacement, on grids of
// up to 1e6 cells per axis), and the pair walk visits every cell next to the
// one a particle is filed in.  (A NaN coordinate converts to 0: cell 0.)
__device__ __forceinline__ int cell_axis(const GridV& v, int k, double x)
{
    const int q = __double2int_rd(__dmul_rn(__dsub_rn(x, v.lo[k]), v.inv_cs[k]));
    return q < 0 ? 0 : (q > v.ncell[k] - 1 ? v.ncell[k] - 1 : q);
}

// Separation b - a along axis k with the minimum-image rule (same operations
// as the oracle).
__device__ __forceinline__ double sep_axis(const GridV& v, int k, double xa, double xb)
{
    double d = __dsub_rn(xb, xa);
    if (v.periodic[k]) {
        double half = __dmul_rn(0.5, v.L[k]);
        if (d > half) d = __dsub_rn(d, v.L[k]);
        else if (d < -half) d = __dadd_rn(d, v.L[k]);
    }
    return d;
}

template <int DIM>
__device__ __forceinline__ bool pair_touches(const GridV& v, double delta, const double* xa, double ra,
                                             const double* __restrict__ pos, const double* __restrict__ radius, int b)
{
    double d2 = 0.0;
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        double d = sep_axis(v, k, xa[k], pos[b * DIM + k]);
        double dd = __dmul_rn(d, d);
        d2 = (k == 0) ? dd : __dadd_rn(d2, dd);
    }
    double s = __dadd_rn(__dadd_rn(ra, radius[b]), delta);
    return d2 < __dmul_rn(s, s);
}

// Single-precision pre-filter of the pair test: true only if the pair is
// certainly not a contact, so that the exact FP64 test above (which alone
// decides) runs only for the candidates that may be.  Each coordinate
// rounded to float is within 2^-24 |x| of the double, so the float
// separation of an axis is within e_k = 2^-23 (|x_a| + |x_b| (+ L on a
// periodic axis)) of the exact one (a factor two over the rounding of the
// conversions, the subtraction and the image shift), and the distance
// within E = sum_k e_k.  A contact has |d| < s, hence a float distance
// below s + E; the relative roundings of d2, of s and of the threshold
// itself are covered by the factors 1 + 2^-20.  An image chosen differently
// near |d| = L/2 changes nothing: a periodic axis spans at least three cells,
// so both images are farther apart than any contact distance.  Squares below
// 2^-126 are rounded to multiples of 2^-149 instead, at most three of them: the
// 2^-126 added to the threshold covers those (lengths below 1e-19; larger squares
// than FP32 has are infinite on both sides, or far).
template <int DIM>
__device__ __forceinline__ bool pair_far_f32(const GridV& v, const float (&Lf)[3], float delta_f, const float4& pa,
                                             const float4& pb)
{
    const float xa[3] = {pa.x, pa.y, pa.z}, xb[3] = {pb.x, pb.y, pb.z};
    float d2 = 0.0f, E = 0.0f;
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        float d = xb[k] - xa[k];
        float m = fabsf(xa[k]) + fabsf(xb[k]);
        if (v.periodic[k]) {
            const float half = 0.5f * Lf[k];
            if (d > half) d -= Lf[k];
            else if (d < -half) d += Lf[k];
            m += Lf[k];
        }
        d2 = fmaf(d, d, d2);
        E = fmaf(m, 1.1920929e-7f, E);   // 2^-23
    }
    const float s = pa.w + pb.w + delta_f;
    const float t = fmaf(s, 1.0f + 9.5367432e-7f, E) * (1.0f + 9.5367432e-7f);   // 1 + 2^-20
    return d2 > fmaf(t, t, 1.1754944e-38f);   // 2^-126
}

// Gap of the particle at xa to wall k (k = 2 axis + side).  The coordinate is
// picked by selects, not by indexing xa with k (a run-time index would put
// the caller's small arrays in local memory).
__device__ __forceinline__ double wall_gap(const double* xa, double ra, const double* wall_pos, int k)
{
    const int axis = k >> 1;
    const double x = (axis == 0) ? xa[0] : (axis == 1) ? xa[1] : xa[2];
    if ((k & 1) == 0) return __dsub_rn(__dsub_rn(x, wall_pos[k]), ra);
    return __dsub_rn(__dsub_rn(wall_pos[k], x), ra);
}

__device__ __forceinline__ bool wall_on(const GridV& v, int dim, int k)
{
    return ((v.wall_mask >> k) & 1) && (k >> 1) < dim;
}

// Walls in contact with the particle at xa (bit k: wall k has gap < delta).
template <int DIM>
__device__ __forceinline__ unsigned wall_mask_of(const CdGeom& g, const GridV& v, const double* wp, const double* xa,
                                                 double ra)
{
    unsigned m = 0u;
#pragma unroll
    for (int k = 0; k < 2 * DIM; ++k)
        if (wall_on(v, DIM, k) && wall_gap(xa, ra, wp, k) < g.delta) m |= 1u << k;
    return m;
}

// Visits the candidate partners b > a of particle a in the 3^DIM cells around
// it (in a's packing grid); calls f(b) for each b that passes the pair test.
// Needs each cell's list sorted by id (k_cell_sort).
//
// The three cells x-1, x, x+1 of one row of the stencil are consecutive cell
// ids, so their particles are one run of cell_pid: 3^(DIM-1) runs (a periodic
// x axis that wraps adds the wrapped cell as a run of its own).  A cell whose
// last id is not above a holds no partner: such cells are trimmed off the
// left end of a run, and a run none of whose cells passes is dropped (ids
// follow the packing's rows, so that is most runs below a's row).  The
// candidates of the runs are then walked as one flat sequence, so the lanes
// of a warp loop about as many times as their own candidate counts.  The
// runs' bounds live in registers (RUNS fixed, the loops unrolled, the next
// run picked by comparisons against compile-time indices): an array of cell
// ranges indexed in a loop went to local memory and dominated the kernel's
// memory traffic.
template <int DIM>
struct Runs {
    static constexpr int N = (DIM == 3) ? 18 : 6;   // 3^(DIM-1) rows, each with a possible wrapped cell
    int lo[N], hi[N];
    // r is a compile-time index at every call (unrolled loops)
    __device__ __forceinline__ void set(int r, int l, int h) { lo[r] = l; hi[r] = h; }
    __device__ __forceinline__ void get(int j, int& l, int& h) const
    {
#pragma unroll
        for (int k = 0; k < N; ++k)
            if (k == j) { l = lo[k]; h = hi[k]; }
    }
};

// The same runs in shared memory, [run][thread] (a warp's accesses fall in
// distinct banks): the counting pass keeps its registers for the walk
// itself, and a run is fetched by its run-time index.
template <int DIM, int STRIDE>
struct RunsShared {
    static constexpr int N = Runs<DIM>::N;
    int* lo;   // &s_lo[0][threadIdx.x], stride STRIDE (the threads of the block)
    int* hi;
    __device__ __forceinline__ void set(int r, int l, int h) { lo[r * STRIDE] = l; hi[r * STRIDE] = h; }
    __device__ __forceinline__ void get(int j, int& l, int& h) const { l = lo[j * STRIDE]; h = hi[j * STRIDE]; }
};

template <typename START>
__device__ __forceinline__ int last_id(const START& cell_start, const int* __restrict__ cell_pid, int cc)
{
    const int l = cell_start[cc], h = cell_start[cc + 1];
    return (h > l) ? cell_pid[h - 1] : -1;
}

// Builds the runs of particle a in R (Runs or RunsShared); the walk starts
// at run 0.  cell_start[c]: first entry of cell c's list (an array, or an
// object that looks it up).  Without SORTED the lists are in no order and
// whole runs are taken.
template <int DIM, bool SORTED, typename RS, typename START>
__device__ __forceinline__ void walk_init(const GridV& v, int a, const int* __restrict__ cell_of,
                                          const START& cell_start, const int* __restrict__ cell_pid, RS& R)
{
    const int c = cell_of[a] - v.base;
    const int n0 = v.ncell[0], n1 = v.ncell[1];
    const int q0 = c % n0;
    const int q1 = (c / n0) % n1;
    const int q2 = c / (n0 * n1);
    const int x0 = (q0 > 0) ? q0 - 1 : 0, x1 = (q0 < n0 - 1) ? q0 + 1 : n0 - 1;
    int xw = -1;   // a periodic x axis: the wrapped neighbour cell outside [x0, x1]
    if (v.periodic[0] && n0 >= 3) {
        if (q0 == 0) xw = n0 - 1;
        else if (q0 == n0 - 1) xw = 0;
    }
    constexpr int ZN = (DIM == 3) ? 3 : 1;
#pragma unroll
    for (int iz = 0; iz < ZN; ++iz) {
#pragma unroll
        for (int iy = 0; iy < 3; ++iy) {
            const int r = 2 * (iz * 3 + iy);
            int l0 = 0, h0 = 0, l1 = 0, h1 = 0;
            int t2 = (DIM == 3) ? q2 + iz - 1 : 0;
            if (DIM == 3 && (t2 < 0 || t2 >= v.ncell[2])) {
                if (!v.periodic[2]) { R.set(r, 0, 0); R.set(r + 1, 0, 0); continue; }
                t2 = (t2 + v.ncell[2]) % v.ncell[2];
            }
            int t1 = q1 + iy - 1;
            if (t1 < 0 || t1 >= n1) {
                if (!v.periodic[1]) { R.set(r, 0, 0); R.set(r + 1, 0, 0); continue; }
                t1 = (t1 + n1) % n1;
            }
            const int row = v.base + (t2 * n1 + t1) * n0;
            if constexpr (!SORTED) {
                l0 = cell_start[row + x0];
                h0 = cell_start[row + x1 + 1];
                if (xw >= 0) {
                    l1 = cell_start[row + xw];
                    h1 = cell_start[row + xw + 1];
                }
                R.set(r, l0, h0);
                R.set(r + 1, l1, h1);
                continue;
            }
            // the run's cells x0 .. x1 (one to three): their bounds, then their last
            // ids (independent loads); the run starts at its first cell with an id above a
            const int nx = x1 - x0 + 1;
            const int cs0 = cell_start[row + x0];
            const int cs1 = (nx > 1) ? cell_start[row + x0 + 1] : 0;
            const int cs2 = (nx > 2) ? cell_start[row + x0 + 2] : 0;
            const int cs3 = cell_start[row + x1 + 1];
            const int e0 = (nx > 1) ? cs1 : cs3, e1 = (nx > 2) ? cs2 : cs3;
            const int L0 = (e0 > cs0) ? cell_pid[e0 - 1] : -1;
            const int L1 = (nx > 1 && e1 > cs1) ? cell_pid[e1 - 1] : -1;
            const int L2 = (nx > 2 && cs3 > cs2) ? cell_pid[cs3 - 1] : -1;
            const int start = (L0 > a) ? cs0 : (L1 > a) ? cs1 : (L2 > a) ? cs2 : -1;
            if (start >= 0) {
                l0 = start;
                h0 = cs3;
            }
            if (xw >= 0 && last_id(cell_start, cell_pid, row + xw) > a) {
                l1 = cell_start[row + xw];
                h1 = cell_start[row + xw + 1];
            }
            R.set(r, l0, h0);
            R.set(r + 1, l1, h1);
        }
    }
}

// The next candidate of the flat walk over the runs (j the run, [s, e) what
// is left of it): its place in the cell lists, or -1 once they are exhausted
// (and on every later call).
template <int DIM, typename RS>
__device__ __forceinline__ int walk_next(const RS& R, int& j, int& s, int& e)
{
    while (s >= e) {
        if (++j >= Runs<DIM>::N) return -1;
        R.get(j, s, e);
    }
    return s++;
}

template <int DIM, bool SORTED, typename START, typename F>
__device__ __forceinline__ void for_each_partner(const CdGeom& g, const GridV& v, int a, const double* xa, double ra,
                                                 const double* __restrict__ pos, const double* __restrict__ radius,
                                                 const int* __restrict__ cell_of, const START& cell_start,
                                                 const int* __restrict__ cell_pid, const float4* __restrict__ pf, F f)
{
    Runs<DIM> R;
    walk_init<DIM, SORTED>(v, a, cell_of, cell_start, cell_pid, R);
    int j = 0, s = R.lo[0], e = R.hi[0];
    // the pre-filter's data (pf null: the exact test only)
    float4 pa = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    const float Lf[3] = {(float)v.L[0], (float)v.L[1], (float)v.L[2]};
    const float delta_f = (float)g.delta;
    if (pf) pa = pf[a];
    for (;;) {
        const int at = walk_next<DIM>(R, j, s, e);
        if (at < 0) break;
        const int b = cell_pid[at];
        if (b > a && !(pf && pair_far_f32<DIM>(v, Lf, delta_f, pa, pf[b])) &&
            pair_touches<DIM>(v, g.delta, xa, ra, pos, radius, b))
            f(b);
    }
}

// Exact tests of the first `take` queued pairs of a warp, lane q on pair q:
// the owner lane's particle (its id, position and radius by shuffles), the
// partner's from memory.  A pair that touches counts for its owner and is
// kept among the owner's first CD_CAND partners.
template <int DIM>
__device__ __forceinline__ void exact_batch(const CdGeom& g, const CdWork& w, const double* __restrict__ pos,
                                            const double* __restrict__ radius, int a, double x0, double x1,
                                            double x2, double ra, int take, const int* qb, const int* qo, int* cnt)
{
    const int lane = threadIdx.x & 31;
    const int o = (lane < take) ? qo[lane] : 0;
    const int b = (lane < take) ? qb[lane] : 0;
    const int ao = __shfl_sync(0xffffffffu, a, o);
    double xo[3];
    xo[0] = __shfl_sync(0xffffffffu, x0, o);
    xo[1] = __shfl_sync(0xffffffffu, x1, o);
    xo[2] = (DIM == 3) ? __shfl_sync(0xffffffffu, x2, o) : 0.0;
    const double ro = __shfl_sync(0xffffffffu, ra, o);
    if (lane < take) {
        GridV vo;
        grid_of(g, w, ao, vo);
        if (pair_touches<DIM>(vo, g.delta, xo, ro, pos, radius, b)) {
            const int slot = atomicAdd(&cnt[o], 1);
            if (w.cand && slot < CD_CAND) w.cand[(size_t)ao * CD_CAND + slot] = b;
        }
    }
}

// Geometry of contact (a, b): normal from a to b, gap, m_n = 1/w_n and
// m_t = 1/w_t with w_n = 1/m_a + 1/m_b, w_t = w_n + r_a^2/I_a + r_b^2/I_b.
// A wall is body n + 6 * packing + k.
template <int DIM>
__device__ __forceinline__ void contact_geometry(const CdGeom& g, const CdWork& w, int a, int b,
                                                 const double* __restrict__ pos, const double* __restrict__ radius,
                                                 const double* __restrict__ inv_m, const double* __restrict__ inv_I,
                                                 double nv[3], double* gap, double* mn, double* mt)
{
    GridV v;
    grid_of(g, w, a, v);
    double xa[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < DIM; ++k) xa[k] = pos[a * DIM + k];
    double ra = radius[a];
    double wa_m = inv_m[a], wa_I = g.rotations ? inv_I[a] : 0.0;
    double wb_m = 0.0, wb_I = 0.0, rb = 0.0;
    nv[0] = nv[1] = nv[2] = 0.0;
    if (b < g.n) {
        double dv[3] = {0.0, 0.0, 0.0};
        double d2 = 0.0;
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            dv[k] = sep_axis(v, k, xa[k], pos[b * DIM + k]);
            double dd = __dmul_rn(dv[k], dv[k]);
            d2 = (k == 0) ? dd : __dadd_rn(d2, dd);
        }
        double d = __dsqrt_rn(d2);
        if (d > 0.0) {
#pragma unroll
            for (int k = 0; k < DIM; ++k) nv[k] = __ddiv_rn(dv[k], d);
        } else {
            nv[0] = 1.0;
        }
        rb = radius[b];
        *gap = __dsub_rn(d, __dadd_rn(ra, rb));
        wb_m = inv_m[b];
        wb_I = g.rotations ? inv_I[b] : 0.0;
    } else {
        int t = b - g.n;
        int k = t % 6;
        const double sgn = (k & 1) ? 1.0 : -1.0;
        const int axis = k >> 1;
        nv[0] = (axis == 0) ? sgn : 0.0;
        nv[1] = (axis == 1) ? sgn : 0.0;
        nv[2] = (axis == 2) ? sgn : 0.0;
        *gap = wall_gap(xa, ra, w.pk_wall_pos + 6 * (t / 6), k);
        // a force-controlled wall moves along its normal only: its inverse
        // mass enters the normal row, not the tangential one
        if (cd_is_body(g, b)) wb_m = g.wall_im[k];
    }
    double w_n = __dadd_rn(wa_m, wb_m);
    double w_t = __dadd_rn(__dadd_rn((b < g.n) ? w_n : wa_m, __dmul_rn(__dmul_rn(ra, ra), wa_I)),
                           __dmul_rn(__dmul_rn(rb, rb), wb_I));
    *mn = (w_n > 0.0) ? __ddiv_rn(1.0, w_n) : 0.0;
    *mt = (w_t > 0.0) ? __ddiv_rn(1.0, w_t) : 0.0;
}

// Files particle i: its cell, the cell's count, and its single-precision copy.
template <int DIM>
__device__ __forceinline__ void count_cell(const CdGeom& g, const CdWork& w, const double* __restrict__ pos,
                                           const double* __restrict__ radius, int i, int* __restrict__ cell_of,
                                           int* __restrict__ cell_cnt)
{
    GridV v;
    grid_of(g, w, i, v);
    if (w.pf) {
        // single-precision copy of (x, y, z, r) for the pair pre-filter
        w.pf[i] = make_float4((float)pos[i * DIM + 0], (float)pos[i * DIM + 1],
                              DIM == 3 ? (float)pos[i * DIM + 2] : 0.0f, (float)radius[i]);
    }
    int c0 = cell_axis(v, 0, pos[i * DIM + 0]);
    int c1 = cell_axis(v, 1, pos[i * DIM + 1]);
    int c2 = (DIM == 3) ? cell_axis(v, 2, pos[i * DIM + 2]) : 0;
    int c = v.base + (c2 * v.ncell[1] + c1) * v.ncell[0] + c0;
    cell_of[i] = c;
    atomicAdd(&cell_cnt[c], 1);
}

// Counting pass: partners b > a of every particle, and its walls.  A lane
// walks its particle's candidates through the single-precision pre-filter;
// the candidates that pass are queued per warp (ballot and prefix count) and
// the warp runs the exact FP64 test on 32 queued pairs at a time, whoever
// owns them.  With the test inside the walk the warp issued it in nearly
// every step, since some lane's candidate nearly always passes the
// pre-filter (~220 FP64 warp instructions per particle warp on the
// 1e6-sphere gas).  The partners found and their count are those of the
// walk; only the order in which a particle's first CD_CAND partners are kept
// depends on timing, and the emitting pass sorts them.  The runs live in
// shared memory and the walk's state in registers: 64 registers, four
// blocks per SM without spills.  The particle's wall contacts are kept as a
// bit mask for the emitting pass.
// The particles base .. base + 31 below `end`, one warp.  qb, qo: CD_QUEUE
// queued partners (at most 31 left over + CD_WALK each) and their owner lanes; cnt_w: 32
// counts; s_lo, s_hi: runs of the block's STRIDE threads, [run][thread].
template <int DIM, int STRIDE, bool SORTED, typename START>
__device__ __forceinline__ void count_pairs(const CdGeom& g, const CdWork& w, const double* __restrict__ pos,
                                            const double* __restrict__ radius, int base, int end,
                                            const int* __restrict__ cell_of, const START& cell_start,
                                            const int* __restrict__ cell_pid, int* __restrict__ pcnt, int* qb, int* qo,
                                            int* cnt_w, int* s_lo, int* s_hi)
{
    CdCtrl* ctrl = w.ctrl;
    const int lane = threadIdx.x & 31;
    const int a = base + lane;
    const bool act = a < end;
    GridV v;
    double xa[3] = {0.0, 0.0, 0.0};
    double ra = 0.0;
    RunsShared<DIM, STRIDE> R;
    R.lo = s_lo + threadIdx.x;
    R.hi = s_hi + threadIdx.x;
    int j = 0, s = 0, e = 0;
    float4 pa = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    float Lf[3] = {0.0f, 0.0f, 0.0f};
    bool more = act;
    if (act) {
        grid_of(g, w, a, v);
#pragma unroll
        for (int k = 0; k < DIM; ++k) xa[k] = pos[a * DIM + k];
        ra = radius[a];
        walk_init<DIM, SORTED>(v, a, cell_of, cell_start, cell_pid, R);
        R.get(0, s, e);
        if (w.pf) pa = w.pf[a];
#pragma unroll
        for (int k = 0; k < 3; ++k) Lf[k] = (float)v.L[k];
    }
    const float delta_f = (float)g.delta;
    cnt_w[lane] = 0;
    __syncwarp();
    int qn = 0;   // queued pairs (the same in every lane)
    for (;;) {
        // CD_WALK candidates a lane at a time: their ids, then their positions,
        // are in flight together
        int b[CD_WALK];
#pragma unroll
        for (int u = 0; u < CD_WALK; ++u) {
            int at = -1;
            if (more) {
                at = walk_next<DIM>(R, j, s, e);
                more = at >= 0;
            }
            b[u] = at;
        }
#pragma unroll
        for (int u = 0; u < CD_WALK; ++u) b[u] = (b[u] >= 0) ? cell_pid[b[u]] : -1;
        bool q[CD_WALK];
        if (w.pf) {
            float4 pb[CD_WALK];
#pragma unroll
            for (int u = 0; u < CD_WALK; ++u)
                if (b[u] > a) pb[u] = w.pf[b[u]];
#pragma unroll
            for (int u = 0; u < CD_WALK; ++u)
                q[u] = act && b[u] > a && !pair_far_f32<DIM>(v, Lf, delta_f, pa, pb[u]);
        } else {
#pragma unroll
            for (int u = 0; u < CD_WALK; ++u) q[u] = act && b[u] > a;
        }
#pragma unroll
        for (int u = 0; u < CD_WALK; ++u) {
            const unsigned m = __ballot_sync(0xffffffffu, q[u]);
            if (q[u]) {
                const int at = qn + __popc(m & ((1u << lane) - 1u));
                qb[at] = b[u];
                qo[at] = lane;
            }
            qn += __popc(m);
        }
        const bool done = !__any_sync(0xffffffffu, more);
        while (qn >= 32 || (done && qn > 0)) {
            __syncwarp();
            const int take = qn < 32 ? qn : 32;
            exact_batch<DIM>(g, w, pos, radius, a, xa[0], xa[1], xa[2], ra, take, qb, qo, cnt_w);
            // the rest to the front of the queue
            const int rest = qn - take;
            for (int r0 = 0; r0 < rest; r0 += 32) {
                int rb = 0, ro = 0;
                if (r0 + lane < rest) { rb = qb[r0 + 32 + lane]; ro = qo[r0 + 32 + lane]; }
                __syncwarp();
                if (r0 + lane < rest) { qb[r0 + lane] = rb; qo[r0 + lane] = ro; }
                __syncwarp();
            }
            qn = rest;
        }
        if (done) break;
    }
    __syncwarp();
    if (act) {
        const int cnt = cnt_w[lane];
        const unsigned wm = wall_mask_of<DIM>(g, v, w.pk_wall_pos + 6 * v.pkid, xa, ra);
        if (w.wmask) w.wmask[a] = (unsigned char)wm;   // the emitting pass reuses it
        if (cnt > CD_MAXLOC) atomicCAS(&ctrl->error, CDE_NONE, CDE_PER_PARTICLE);
        pcnt[a] = cnt + __popc(wm);
    }
    __syncwarp();
}

// Emitting pass: the keys (a, b) of every particle's contacts, partners in
// ascending id, then its walls, at the particle's offset from the scan of
// the counts.  Integer work only; the geometry follows one thread per
// contact (k_geometry_warm).
// Particle a's contacts from position o of the new set on.
template <int DIM, bool SORTED, typename START>
__device__ __forceinline__ void emit_pairs(const CdGeom& g, const CdWork& w, const double* __restrict__ pos,
                                           const double* __restrict__ radius, int a, int o, const START& cell_start)
{
    GridV v;
    grid_of(g, w, a, v);
    double xa[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < DIM; ++k) xa[k] = pos[a * DIM + k];
    double ra = radius[a];
    // the counting pass's walls (the same test, so not repeated in FP64)
    const unsigned wm = w.wmask ? (unsigned)w.wmask[a]
                                : wall_mask_of<DIM>(g, v, w.pk_wall_pos + 6 * v.pkid, xa, ra);
    const int npart = w.pcnt[a] - __popc(wm);   // partners the counting pass found
    if (w.cand && npart <= CD_CAND) {
        // the counting pass kept them (in the order its exact tests ran):
        // emit in ascending id by repeated selection of the smallest one
        // above the last emitted
        const int* keep = w.cand + (size_t)a * CD_CAND;
        int last = a;
        for (int f = 0; f < npart; ++f) {
            int bmin = INT_MAX;
            for (int q = 0; q < npart; ++q) {
                const int bq = keep[q];
                if (bq > last && bq < bmin) bmin = bq;
            }
            w.pairs_nx[o++] = make_int2(a, bmin);
            last = bmin;
        }
    } else {
        int found[CD_MAXLOC];
        int nf = 0;
        auto insert = [&](int b) {
            if (nf < CD_MAXLOC) {
                // insertion into the sorted prefix
                int j = nf++;
                while (j > 0 && found[j - 1] > b) { found[j] = found[j - 1]; --j; }
                found[j] = b;
            }
        };
        for_each_partner<DIM, SORTED>(g, v, a, xa, ra, pos, radius, w.cell_of, cell_start, w.cell_pid, w.pf, insert);
        for (int f = 0; f < nf; ++f) w.pairs_nx[o++] = make_int2(a, found[f]);
    }
#pragma unroll
    for (int k = 0; k < 2 * DIM; ++k)
        if ((wm >> k) & 1u) w.pairs_nx[o++] = make_int2(a, g.n + 6 * v.pkid + k);
}

// Geometry of every detected contact, one thread per contact (so that the
// FP64 square root and divisions run on full warps), and its starting
// impulse: matched by key in the current (previous) set; in 3D the old
// tangential impulse is projected onto the new tangent plane.
// nold: contacts of the previous set; by_particle: its per-particle offsets
// are kept (poff_prev).
template <int DIM>
__device__ __forceinline__ void geometry_warm(const CdGeom& g, const CdWork& w, int c, int nold, int by_particle,
                                              const double* __restrict__ pos, const double* __restrict__ radius,
                                              const double* __restrict__ inv_m, const double* __restrict__ inv_I,
                                              int warm, int pw)
{
    const int2 ab = w.pairs_nx[c];
    double nv[3], gap, mn, mt;
    contact_geometry<DIM>(g, w, ab.x, ab.y, pos, radius, inv_m, inv_I, nv, &gap, &mn, &mt);
    w.nrm[3 * c + 0] = nv[0];
    w.nrm[3 * c + 1] = nv[1];
    w.nrm[3 * c + 2] = nv[2];
    w.gap[c] = gap;
    w.mn[c] = mn;
    w.mt[c] = mt;
    double out[4] = {0.0, 0.0, 0.0, 0.0};
    if (warm && nold > 0) {
        const unsigned long long key = cd_key(ab.x, ab.y);
        // the old set is in key order, so particle a's old contacts are the
        // range its offsets give (when kept), else somewhere in the whole set
        int lo = 0, hi = nold - 1, o = -1;
        if (by_particle) {
            lo = w.poff_prev[ab.x];
            hi = w.poff_prev[ab.x + 1] - 1;
        }
        while (lo <= hi) {
            int mid = lo + ((hi - lo) >> 1);
            int2 m = w.pairs[mid];
            unsigned long long km = cd_key(m.x, m.y);
            if (km == key) { o = mid; break; }
            if (km < key) lo = mid + 1; else hi = mid - 1;
        }
        if (o >= 0) {
            if (DIM == 2) {
                out[0] = w.Pk[2 * o];
                out[1] = w.Pk[2 * o + 1];
            } else {
                const double* q = w.Pk + 4 * o;
                double tn = __dadd_rn(__dadd_rn(__dmul_rn(q[1], nv[0]), __dmul_rn(q[2], nv[1])),
                                      __dmul_rn(q[3], nv[2]));
                out[0] = q[0];
                out[1] = __dsub_rn(q[1], __dmul_rn(tn, nv[0]));
                out[2] = __dsub_rn(q[2], __dmul_rn(tn, nv[1]));
                out[3] = __dsub_rn(q[3], __dmul_rn(tn, nv[2]));
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (k < pw) w.Pk_nx[pw * c + k] = out[k];   // compile-time indices keep out[] in registers
}
