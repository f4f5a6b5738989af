// cd_flow.cu -- the impulse solve as a dataflow over the contacts (plain
// systems, their domain-wise update, batches): the colour order without a grid
// barrier per colour.
//
// The colour order says, for every body, in which order its contacts update
// it.  Nothing else orders the updates: an update may run as soon as both its
// bodies have had all their earlier ones.  So every body's velocity record
// carries the number of updates it has had, and a warp (32 contacts of one
// colour; the block's warps take the block's contacts colour by colour) looks
// at its bodies' records until they carry the numbers it expects.  The blocks
// are all resident (cooperative launch) and every warp takes its items in
// colour order, so the earliest item not yet done can always run: no wait is
// circular, and each is bounded as well.  The bits are those of the barrier
// schedule.
//
// A block keeps its contacts' records (impulse included) in shared memory for
// the whole solve where they fit; a system too large for that reads them
// through L1.  One more warp takes the block's residual terms, publishes their
// sum, gathers the other blocks' and runs the convergence test.  That stays off
// the path: after the first sweeps a sweep starts before the
// test of the one (then two) before it is known.  The impulses of the last
// three sweeps are kept in turn, and the velocities from before the last two,
// so the sweeps begun past the last one are taken back.
//
// What bounds it: in FP64 the FP64 pipe (64 cycles a warp instruction on each
// quarter of an SM, 25 of them a warp of contacts: ~3,200 cycles a colour of the
// 100,000-disc pile) and then the way of the records to the next colour (~1,700)
// in turn, since neighbouring blocks move in step; in FP32, and in small systems, the way of a record
// from SM to SM (~500 cycles on a die, ~850 across) once per colour, plus the
// update (FP64: ~1,700 cycles for a whole warp of contacts; ~1,100 for 16
// contacts split over lane pairs, where a block has few).  Per sweep, against
// the barrier schedule (grid barrier 2,900 cycles a colour, then the velocity
// loads): 100,000-disc pile FP64 28.4 -> 17.3 us, FP32 18.0 -> 9.5 us;
// 5,000 discs FP64 20.6 -> 9.7 us; 2,000 discs 18.0 -> 8.3 us.  Tried and not kept: one lane
// looking for its warp (FP32 7% slower, 5,000 discs 12%), pauses between looks
// (5,000 discs 2 to 15% slower), 15 or 7 updating warps in place of 11 (FP64 2
// and 17% slower), records through L1 (FP64 pile 24.3 us a sweep), two far-apart
// regions a block on four warps each, to run one while the other waits (they
// fall into step: FP64 10% slower, FP32 19%).
#include "cd_flow_core.cuh"
#include "cd_pack_core.cuh"

#define FLOW_WORKERS 11                           // warps that update contacts
#define FLOW_THREADS (32 * (FLOW_WORKERS + 1))    // and one that runs the convergence test
#define FLOW_TAIL 4                               // rounds of packings left from which teams are cut whatever is left over
#define FLOW_LEAST 112                            // contacts that a block of a batched system is given at least
#define FLOW_ROWS 8                               // rows of tagged block sums: while a block leaves those of pass p
                                                  // another may still wait for those of p - 5
#define FLOW_SLOTS 4                              // passes whose residual terms are kept
#define FLOW_LAG1 16                              // from this pass on one starts before the test of the one before is
#define FLOW_LAG2 32                              // known, from this one on two do: what they change can be taken back
// FP64 2D: a block's contacts of a colour up to which two lanes share one.  At 64
// the pairs fill four warps, one for each of the SM's FP64 quarters, 14
// instructions deep in place of two warps 24 deep; beyond, a quarter would
// take two warps of 14, more than one of 24.
#define FLOW_SPLIT 64

// The blocks that solve a system (or a packing) together: nb of the grid from
// block `start` on, this one the blk-th, with a barrier word of their own.  The
// first `work` of them have contacts; the others take part in the tests only.
struct FlowTeam {
    unsigned* word;
    int start, nb, blk, work;
    __device__ __forceinline__ bool sync(CdCtrl* ctrl) const
    {
        if (nb == 1) {
            __syncthreads();
            return true;
        }
        return cd_team_sync(ctrl, word, (unsigned)nb, blk == 0);
    }
};

#define FLOW_KINDS (CD_KMAX + 1)

// What the block's warps share.
struct FlowShared {
    // by colour (and the shared particles' sums as one more)
    int lo[FLOW_KINDS], end[FLOW_KINDS];   // this block's positions
    int half[FLOW_KINDS];                  // 1: its contacts are split over two lanes each
    int base[FLOW_KINDS + 1];              // first of its warp items (32 contacts, or 16 split over two lanes each)
    int slot[FLOW_KINDS + 1];              // contacts of the colours before: place in the block's records
    int before[FLOW_KINDS];                // the colour with items before each (in turn), or -1 - the last one
    int done[FLOW_KINDS];                  // its warp items done, over all passes
    double acc[FLOW_SLOTS][FLOW_WORKERS][32]; // residual terms of a pass by worker lane
    int arrived[FLOW_SLOTS];         // workers that have left them (counted over the passes of a slot)
    int decided;                     // last pass the test is known of
    int stop;                        // the sweep the iteration ends with, once known (else -1)
    int dead;                        // a wait gave up
    double ravg, resid;
    int converged;
};

// Waits in shared memory until *p >= v; false when a wait gave up.
__device__ __forceinline__ bool flow_wait_shared(CdCtrl* ctrl, FlowShared& sh, const int* p, int v)
{
    FlowBound bound;
    while (flow_ld(p) < v) {
        if (flow_ld(&sh.dead)) return false;
        if (!bound.go(ctrl)) {
            *(volatile int*)&sh.dead = 1;
            return false;
        }
    }
    __threadfence_block();
    return true;
}

__device__ __forceinline__ double shfl_pair(double v) { return __shfl_xor_sync(0xffffffffu, v, 1); }

// The control warp's state: the next pass whose block sum it leaves, and the
// next one whose test it decides.
struct FlowControl {
    int pub = 0, dec = 0;
    double xprev = 0.0;
};

// The control warp: leaves the block's sum of a pass when the workers have
// finished it, and decides the test of the first undecided pass when every
// block's sum is there (whichever comes first: neither waits for the other).
// Returns after a decision; false when a wait gave up.  Every block adds the same
// sums in the same order, so all decide alike.
__device__ __forceinline__ bool flow_control(CdCtrl* ctrl, FlowShared& sh, FlowSum* part, const FlowTeam& tm,
                                             FlowControl& fc, int nc, int crit, double alpha, int max_sweeps)
{
    const int lane = threadIdx.x & 31;
    const int nb = tm.nb;
    FlowBound bound;
    double x = 0.0;
    for (int b0 = 0; b0 < nb;) {
        if (__all_sync(0xffffffffu, flow_ld(&sh.arrived[fc.pub % FLOW_SLOTS]) >= FLOW_WORKERS * (fc.pub / FLOW_SLOTS + 1))) {
            __threadfence_block();
            __syncwarp();
            double v[FLOW_WORKERS];
#pragma unroll
            for (int u = 0; u < FLOW_WORKERS; ++u)
                v[u] = *(volatile double*)&sh.acc[fc.pub % FLOW_SLOTS][u][lane];
            const double y = flow_sum_warp(v);
            if (lane == 0)
                flow_sum_store(part + (size_t)(fc.pub % FLOW_ROWS) * gridDim.x + tm.start + tm.blk, y,
                               (unsigned)fc.pub + 1u);
            ++fc.pub;
        }
        if (fc.dec < fc.pub && (bound.spins & 3u) == 0u) {   // (looks take bandwidth from the workers')
            // five blocks a lane at a time, their loads in flight together
            const FlowSum* row = part + (size_t)(fc.dec % FLOW_ROWS) * gridDim.x + tm.start;
            u64 f[5][2];
            double v[5];
            bool have = true;
#pragma unroll
            for (int u = 0; u < 5; ++u) {
                const int b = b0 + 32 * u + lane;
                if (b < nb) flow_load(row[b].e, f[u]);
            }
#pragma unroll
            for (int u = 0; u < 5; ++u) {
                const bool in = b0 + 32 * u + lane < nb;
                have = have && (!in || flow_sum_is(f[u], (unsigned)fc.dec + 1u));
                v[u] = in ? flow_sum_of(f[u]) : 0.0;
            }
            if (__all_sync(0xffffffffu, have)) {
                const double y = flow_sum_warp(v);
                x = b0 ? x + y : y;
                b0 += 160;
            }
        }
        if (!__all_sync(0xffffffffu, bound.go(ctrl) && !flow_ld(&sh.dead))) return false;
    }
    const int pass = fc.dec++;
    if (lane == 0) {
        // the ratio of the test against its threshold by products; only where
        // that is within rounding of the threshold (or at the end) the test
        // itself, whose FP64 divisions take longer than the rest
        bool end = pass >= max_sweeps;
        if (pass > 0 && crit != CD_CONV_NONE && !end) {
            const double a = (crit == CD_CONV_GLOBAL_SQ) ? sqrt(alpha) : alpha;
            const double s = x + fc.xprev, off = fabs(x - fc.xprev) - a * s;
            end = !(off > s * (1e-15 * (1.0 + a)));
        }
        if (end) {
            const double ra = x / (double)nc;
            double rs = 0.0;
            int cv = 0;
            if (pass > 0) global_test(ra, fc.xprev / (double)nc, crit, alpha, rs, cv);
            *(volatile double*)&sh.ravg = ra;
            *(volatile double*)&sh.resid = rs;
            *(volatile int*)&sh.converged = cv;
            if (cv || pass >= max_sweeps) *(volatile int*)&sh.stop = pass;
        }
        __threadfence_block();
        *(volatile int*)&sh.decided = pass;
    }
    fc.xprev = x;
    __syncwarp();
    return true;
}

// The block's contact records kept in shared memory for the solve (structure
// of arrays over `cap` contacts): all that an update needs except velocities.
template <int DIM, typename T>
struct FlowRecords {
    typedef typename Vec<T>::V4 T4;
    typedef typename Vec<T>::V2 T2;
    typedef typename std::conditional<DIM == 2, T2, T4>::type TP;    // impulse record
    typedef typename std::conditional<DIM == 2, T, T2>::type TM;     // m_t, or (m_n, m_t)
    static constexpr int BYTES = (int)(sizeof(T4) + sizeof(TP) + 3 * sizeof(T2) + sizeof(TM) + sizeof(int2) +
                                       sizeof(unsigned));
    T4* geo;
    TP* P;
    T2* s0;   // (1/m_a, r_a)
    T2* s1;   // (r_a/I_a, 1/m_b)
    T2* s2;   // (r_b, r_b/I_b)
    TM* m;
    int2* ab;
    unsigned* ord;
    __device__ __forceinline__ FlowRecords(char* base, int cap)
    {
        geo = (T4*)base;
        P = (TP*)(geo + cap);
        s0 = (T2*)(P + cap);
        s1 = s0 + cap;
        s2 = s1 + cap;
        m = (TM*)(s2 + cap);
        ab = (int2*)(m + cap);
        ord = (unsigned*)(ab + cap);
    }
};

// The FP64 2D update of core2d by two lanes a contact: the even one takes the
// normal row and the y components, the odd one the tangential row and the x
// components; the same operations with the same rounding, 14 in a row instead
// of 24.  What differs between the lanes are operands chosen before the
// velocities are there: between two FP64 instructions a select or a shuffle
// costs ~44 cycles beyond their own 64 each.
struct FlowHalf {
    double c1, c2, c3, c4, c5, bias, Pold;
    __device__ __forceinline__ void choose(bool odd, const Rec<2, double>& r)
    {
        c1 = odd ? -r.geo.y : r.geo.x;
        c2 = odd ? r.geo.x : r.geo.y;
        c3 = odd ? -r.sa.y : 1.0;
        c4 = odd ? -r.sb.y : 0.0;
        c5 = odd ? -r.mt : -r.geo.w;
        bias = r.geo.z;
        Pold = odd ? r.P.y : r.P.x;
    }
    // Returns this lane's impulse component, and in v1 the new velocity record
    // of body a (even lane) or b (odd).  wall_k: b - n (>= 0: b is the
    // force-controlled wall wall_k, which moves along its normal only).
    __device__ __forceinline__ double update(bool odd, const Rec<2, double>& r, const Vec<double>::V4& va,
                                             const Vec<double>::V4& vb, int wall_k, bool apply_only,
                                             Vec<double>::V4& v1) const
    {
        const double xa = odd ? va.x : va.y, xb = odd ? vb.x : vb.y;
        double Pnew = Pold, d = Pold;
        if (!apply_only) {
            const double u3 = odd ? va.z : bias, u4 = odd ? vb.z : 0.0;
            const double dvx = __dsub_rn(vb.x, va.x), dvy = __dsub_rn(vb.y, va.y);
            double u = __fma_rn(dvy, c2, __dmul_rn(dvx, c1));     // u_n     | (dv x n)
            u = __fma_rn(c3, u3, u);                              // b + u_n | - r_a w_a
            u = __fma_rn(c4, u4, u);                              //         | - r_b w_b
            const double Ps = __fma_rn(c5, u, Pold);
            const double lim = pos_part(shfl_pair(__dmul_rn(r.mu, Ps)));   // mu max(P_n*, 0)
            Pnew = odd ? clamp_sym(Ps, lim) : pos_part(Ps);
            d = __dsub_rn(Pnew, Pold);
        }
        const double e = shfl_pair(d);
        const double dPn = odd ? e : d, dPt = odd ? d : e;
        const double dP = __fma_rn(dPn, c2, __dmul_rn(dPt, c1));  // y | x
        const double xa1 = __fma_rn(-r.sa.x, dP, xa);
        double xb1 = __fma_rn(r.sb.x, dP, xb);
        double om = __fma_rn(odd ? -r.sb.z : -r.sa.z, dPt, odd ? vb.z : va.z);   // of this lane's body
        if (wall_k >= 0) {
            if (((wall_k >> 1) == 0) != odd) xb1 = 0.0;
            if (odd) om = 0.0;
        }
        const double other = shfl_pair(odd ? xa1 : xb1);
        v1.x = odd ? xb1 : other;
        v1.y = odd ? other : xa1;
        v1.z = om;
        v1.w = 0.0;
        return Pnew;
    }
};

__device__ __forceinline__ void* flow_impulses(const CdWork& w, int pass)
{
    const int u = pass % 3;
    return u == 0 ? w.c_P : u == 1 ? w.fl_P : w.fl_P2;
}

// Record r of a contact's second body moves: a particle's, a view's or a
// force-controlled wall's, not a kinematic wall's.
template <bool VIEWS>
__device__ __forceinline__ bool flow_moves(const CdGeom& g, int r)
{
    return VIEWS ? (r < g.n || r >= cd_view_base(g)) : cd_is_body(g, r);
}

// 1 if record r belongs to a particle with several.
__device__ __forceinline__ unsigned flow_shared(const CdWork& w, int vbase, int n, int r)
{
    return r >= vbase || (r < n && w.view_off[r + 1] > w.view_off[r]) ? 1u : 0u;
}

// The sums after a pass's contacts (dom_combine's, in its order): a lane for
// each view, the particle's first one works.
template <int DIM, typename T>
__device__ __forceinline__ bool flow_sum_views(const CdGeom& g, const CdWork& w, CdCtrl* ctrl, FlowShared& sh, u64* VT,
                                               int vbase, int q, bool act, int pass)
{
    typedef FlowBody<DIM, T> Body;
    typedef typename Vec<T>::V4 T4;
    constexpr int EB = Body::G * Body::N;
    constexpr int RW = (DIM == 2) ? 1 : 2;
    T4* V0 = (T4*)w.V0;
    const int i = act ? w.view_owner[q] : 0;
    const bool lead = act && q == w.view_off[i];
    const int e = lead ? w.view_off[i + 1] : q;
    const unsigned ni = lead ? (unsigned)__popcll(w.fl_mask[i]) : 0u;
    FlowBound bound;
    bool ready = !lead;
    while (!__all_sync(0xffffffffu, ready)) {
        if (!ready) {
            Body x;
            x.load(VT + (size_t)EB * i);
            ready = x.has((unsigned)pass * (ni + 1u) + ni);
            for (int u = q; u < e && ready; ++u) {
                const unsigned nu = (unsigned)__popcll(w.fl_mask[vbase + u]);
                x.load(VT + (size_t)EB * (vbase + u));
                ready = x.has((unsigned)pass * (nu + 1u) + nu);
            }
        }
        if ((++bound.spins & 63u) == 0u && !__all_sync(0xffffffffu, bound.look(ctrl) && !flow_ld(&sh.dead))) {
            *(volatile int*)&sh.dead = 1;
            return false;
        }
    }
    if (lead) {
        Body x;
        T4 v, o, a, b, s0 = V0[RW * q], o0 = s0;
        x.load(VT + (size_t)EB * i);
        x.unpack(v, o);
        v.x = s0.x + (v.x - s0.x); v.y = s0.y + (v.y - s0.y); v.z = s0.z + (v.z - s0.z);
        if constexpr (DIM == 3) {
            o0 = V0[RW * q + 1];
            o.x = o0.x + (o.x - o0.x); o.y = o0.y + (o.y - o0.y); o.z = o0.z + (o.z - o0.z);
        }
        for (int u = q; u < e; ++u) {
            x.load(VT + (size_t)EB * (vbase + u));
            x.unpack(a, b);
            v.x = v.x + (a.x - s0.x); v.y = v.y + (a.y - s0.y); v.z = v.z + (a.z - s0.z);
            if constexpr (DIM == 3) {
                o.x = o.x + (b.x - o0.x); o.y = o.y + (b.y - o0.y); o.z = o.z + (b.z - o0.z);
            }
        }
        V0[RW * q] = v;
        if constexpr (DIM == 3) V0[RW * q + 1] = o;
        x.pack(v, o, (unsigned)(pass + 1) * (ni + 1u));
        x.store(VT + (size_t)EB * i);
        for (int u = q; u < e; ++u) {
            x.pack(v, o, (unsigned)(pass + 1) * ((unsigned)__popcll(w.fl_mask[vbase + u]) + 1u));
            x.store(VT + (size_t)EB * (vbase + u));
        }
    }
    __syncwarp();
    return true;
}

// Contact r, open before the update, stays open.
template <typename T>
__device__ __forceinline__ bool flow_stays_open(const Rec<2, T>& r, const typename Vec<T>::V4& va,
                                                const typename Vec<T>::V4&, const typename Vec<T>::V4& vb,
                                                const typename Vec<T>::V4&)
{
    // (FP64 takes an undefined tangential impulse as 0)
    if (sizeof(T) == 4 && !(tame<T>(exponent_of(va.z), exponent_of(r.sa.y)) &&
                            tame<T>(exponent_of(vb.z), exponent_of(r.sb.y)))) return false;
    return stays_open<T>(r.geo.w, gap_rate2d<T>(r.geo.x, r.geo.y, r.geo.z, sub_of<T>(vb.x, va.x),
                                                sub_of<T>(vb.y, va.y)));
}
template <typename T>
__device__ __forceinline__ bool flow_stays_open(const Rec<3, T>& r, const typename Vec<T>::V4& va,
                                                const typename Vec<T>::V4& wa, const typename Vec<T>::V4& vb,
                                                const typename Vec<T>::V4& wb)
{
    T gx, gy, gz;
    const T un = contact_velocity3d<T>(r, va, wa, vb, wb, gx, gy, gz);
    return tame<T>(max(max(exponent_of(gx), exponent_of(gy)), exponent_of(gz)), exponent_of(r.m.y)) &&
           stays_open<T>(r.m.x, add_of<T>(r.geo.w, un));
}

__device__ __forceinline__ bool flow_zero(double2 P) { return ((__double_as_longlong(P.x) | __double_as_longlong(P.y)) << 1) == 0LL; }
__device__ __forceinline__ bool flow_zero(float2 P) { return P.x == 0.0f && P.y == 0.0f; }
template <typename V>
__device__ __forceinline__ bool flow_zero(const V& P)
{
    if constexpr (sizeof(V) == 32)
        return ((__double_as_longlong(P.x) | __double_as_longlong(P.y) | __double_as_longlong(P.z) |
                 __double_as_longlong(P.w)) << 1) == 0LL;
    else return P.x == 0.0f && P.y == 0.0f && P.z == 0.0f && P.w == 0.0f;
}

// The solve of nc contacts by a team of blocks: K colours, colour k at the
// colour-order positions [sh.lo[k], sh.end[k]) (narrowed to this block's), on
// the particles body0 .. body1 - 1 (and the force-controlled walls).  Leaves
// the velocities in w.V, the impulses in colour order (c_P) or key order (Pk),
// the sweeps and the test in sh.  False when a wait gave up.
//
// VIEWS: the domain-wise update (Sec. 3.1).  Contacts work on the velocity
// records of their domain (c_vab); after a pass's contacts one lane for each
// particle with several records adds up their changes and stores the sum to
// all of them, one more update of each: the sums are a colour after the last.
// (A barrier after each colour and after the sums took 28.9 ms for a step of
// 20,000 discs in 4 x 4 domains at FP64, this 13.2.)
template <int DIM, typename T, bool BATCH, bool VIEWS>
__device__ __forceinline__ bool flow_solve(const CdGeom& g, const CdWork& w, FlowShared& sh, char* s_rec, int rec_cap,
                                           const FlowTeam& tm, const CdState& io, int K, int nc, T mu, int body0, int body1, int crit,
                                           double alpha, int max_sweeps)
{
    typedef FlowBody<DIM, T> Body;
    typedef FlowRecords<DIM, T> Records;
    typedef typename Vec<T>::V4 T4;
    typedef typename Vec<T>::V2 T2;
    typedef typename Records::TP TP;
    typedef typename Records::TM TM;
    constexpr int EB = Body::G * Body::N;   // elements of a body's record
    constexpr bool F64_2D = (DIM == 2) && std::is_same<T, double>::value;
    // |P| of an update is taken while the warp's next one waits (3D FP64 has no registers left for it)
    constexpr bool DEFER = (DIM == 2) || std::is_same<T, float>::value;
    CdCtrl* ctrl = w.ctrl;
    const int nw = tm.work;
    const int tid = tm.blk * blockDim.x + threadIdx.x, stride = tm.nb * blockDim.x;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    u64* VT = (u64*)w.fl_V;
    FlowSum* part = (FlowSum*)w.fl_part;
    T4* V = (T4*)w.V;
    T4* Vprev = (T4*)w.fl_Vprev;
    constexpr int RW = (DIM == 2) ? 1 : 2;
    const int nprev = g.n + 6;                        // records in Vprev (a view is taken back with its particle)
    const int nview = VIEWS && nc > 0 ? w.view_off[g.n] : 0;   // records of the domains past the particles' own
    const int vbase = cd_view_base(g);
    const int KX = VIEWS ? K + 1 : K;

    // this block's positions of each colour, and their warp items
    if (threadIdx.x < 32) {
        int run = 0, srun = 0;
        for (int k0 = 0; k0 < KX; k0 += 32) {
            const int k = k0 + lane;
            int m = 0, c = 0;
            if (k < KX) {
                // whole warp items, dealt so that the blocks' totals over the colours
                // are even: colour k's remainder starts at another block
                const int lo = k < K ? sh.lo[k] : 0, hi = k < K ? sh.end[k] : nview;
                const int half = F64_2D && k < K && hi - lo <= FLOW_SPLIT * nw;
                const int sh_item = half ? 4 : 5;
                const unsigned items = (unsigned)(hi - lo + (1 << sh_item) - 1) >> sh_item;
                const unsigned r = (unsigned)(k * 5 * nw >> 3) % (unsigned)nw;
                const unsigned each = items / (unsigned)nw, rest = items % (unsigned)nw;   // (32-bit: items * nw might not fit)
                const unsigned b = min(tm.blk, nw), e = min(tm.blk + 1, nw);
                const int i0 = (int)(each * b + (rest * b + r) / (unsigned)nw);
                const int i1 = (int)(each * e + (rest * e + r) / (unsigned)nw);
                sh.lo[k] = min(lo + (i0 << sh_item), hi);
                sh.end[k] = min(lo + (i1 << sh_item), hi);
                sh.half[k] = half;
                c = k < K ? sh.end[k] - sh.lo[k] : 0;
                m = i1 - i0;
            }
            int incl = m, ci = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o), z = __shfl_up_sync(0xffffffffu, ci, o);
                if (lane >= o) { incl += y; ci += z; }
            }
            if (k < KX) { sh.base[k + 1] = run + incl; sh.slot[k + 1] = srun + ci; }
            run += __shfl_sync(0xffffffffu, incl, 31);
            srun += __shfl_sync(0xffffffffu, ci, 31);
        }
        if (lane == 0) sh.base[0] = sh.slot[0] = 0;
        __syncwarp();
        if (lane == 0) {
            for (int u = 0; u < FLOW_SLOTS; ++u) sh.arrived[u] = 0;
            int prev = -1;
            for (int k = 0; k < KX; ++k) {
                sh.before[k] = prev;
                sh.done[k] = 0;
                if (sh.base[k + 1] > sh.base[k]) prev = k;
            }
            for (int k = 0; k < KX && sh.before[k] < 0; ++k) sh.before[k] = -1 - prev;
            sh.decided = -1;
            sh.stop = (nc == 0) ? 0 : -1;
            sh.dead = 0;
            sh.ravg = sh.resid = 0.0;
            sh.converged = (nc == 0);
        }
    }
    // tagged records (tag 0), cleared block sums
    for (int i = body0 + tid; i < body1; i += stride) {
        if (!cd_is_body(g, i)) continue;
        Body x;
        T4 o;
        o.x = o.y = o.z = o.w = (T)0;
        if constexpr (DIM == 3) o = V[RW * i + 1];
        x.pack(V[RW * i], o, 0u);
        x.store(VT + (size_t)EB * i);
    }
    if constexpr (VIEWS) {
        T4* V0 = (T4*)w.V0;   // the pass start of each particle with views, by its first view
        for (int q = tid; q < nview; q += stride) {
            const int i = w.view_owner[q];
            Body x;
            T4 o;
            o.x = o.y = o.z = o.w = (T)0;
            if constexpr (DIM == 3) { o = V[RW * i + 1]; V0[RW * q + 1] = o; }
            const T4 v = V[RW * i];
            V0[RW * q] = v;
            x.pack(v, o, 0u);
            x.store(VT + (size_t)EB * (vbase + q));
        }
    }
    if (threadIdx.x < FLOW_ROWS) flow_sum_store(part + threadIdx.x * gridDim.x + blockIdx.x, 0.0, 0u);
    __syncthreads();
    const int Q = sh.base[KX];
    const bool res = sh.slot[K] <= rec_cap;   // the block's records fit its shared memory
    Records rec(s_rec, rec_cap);
    // the colours each body has
    for (int k = 0; k < K; ++k)
        for (int p = sh.lo[k] + (int)threadIdx.x; p < sh.end[k]; p += blockDim.x) {
            const int2 ab = VIEWS ? w.c_vab[p] : w.c_ab[p];   // (a wall's place in c_vab is its own)
            atomicOr(&w.fl_mask[ab.x], 1ULL << k);
            if (flow_moves<VIEWS>(g, ab.y)) atomicOr(&w.fl_mask[ab.y], 1ULL << k);
        }
    if (!tm.sync(ctrl)) return false;
    // a contact's place among each body's contacts and their number (8 bits
    // each), and the resident records
    for (int k = 0; k < K; ++k)
        for (int p = sh.lo[k] + (int)threadIdx.x; p < sh.end[k]; p += blockDim.x) {
            Rec<DIM, T> r;
            r.ab = w.c_ab[p];
            const int2 rr = VIEWS ? w.c_vab[p] : r.ab;   // the bodies' records
            const u64 below = (1ULL << k) - 1ULL;
            const u64 ma = w.fl_mask[rr.x], mb = flow_moves<VIEWS>(g, rr.y) ? w.fl_mask[rr.y] : 0ULL;
            unsigned na = (unsigned)__popcll(ma), nbd = (unsigned)__popcll(mb);
            if constexpr (VIEWS) {   // the sum is an update too
                na += flow_shared(w, vbase, g.n, rr.x);
                if (mb) nbd += flow_shared(w, vbase, g.n, rr.y);
            }
            const unsigned ord = (unsigned)__popcll(ma & below) | (na << 8) | ((unsigned)__popcll(mb & below) << 16) |
                                 (nbd << 24);
            if (res) {
                const int i = sh.slot[k] + p - sh.lo[k];
                load_static<DIM, T>(g, w, r);
                T2 t;
                t.x = r.sa.x; t.y = r.sa.y; rec.s0[i] = t;
                t.x = r.sa.z; t.y = r.sb.x; rec.s1[i] = t;
                t.x = r.sb.y; t.y = r.sb.z; rec.s2[i] = t;
                rec.geo[i] = ((const T4*)w.c_geo)[p];
                rec.m[i] = ((const TM*)w.c_m)[p];
                rec.P[i] = ((const TP*)w.c_P)[p];
                rec.ab[i] = rr;
                rec.ord[i] = ord;
            } else {
                w.fl_ord[p] = ord;
            }
        }
    __syncthreads();

    int last = 0;   // last pass this warp has run
    // FP32: wait for the block's own colour before
    // looking.  The looks that find nothing fill the L1's request queue and hold
    // up everything else there (100,000 discs: 15.4 -> 10.9 us a sweep; 20,000 discs, a
    // warp or none an item: 11.6 -> 9.2; 10,000 spheres on a lattice, 11 contacts each, whose records
    // are twice as long: 72 -> 31, behind barriers 63).  FP64
    // items take longer than that and gain from starting early (100,000 discs gated:
    // 18.7 -> 21.3 us).
    constexpr bool gate = sizeof(T) == 4;
    if (nc > 0 && wid == FLOW_WORKERS) {
        FlowControl fc;
        do {
            if (!flow_control(ctrl, sh, part, tm, fc, nc, crit, alpha, max_sweeps)) {
                *(volatile int*)&sh.dead = 1;
                break;
            }
        } while (flow_ld(&sh.stop) < 0);
    } else if (nc > 0) {
        TP pend;   // impulse of the warp's last update whose magnitude is not summed yet
        for (int pass = 0; ; ++pass) {   // pass 0: the starting impulses; pass s: sweep s
            const bool apply_only = (pass == 0);
            // (pass 0 has no test to wait for)
            const int known = pass - 1 - (pass >= FLOW_LAG1) - (pass >= FLOW_LAG2);
            bool on = known < 1 || flow_wait_shared(ctrl, sh, &sh.decided, known);
            on = on && pass <= max_sweeps && !flow_ld(&sh.dead);
            // (a stop after `known` is not looked at: every warp of the grid runs the same passes)
            if (on) {
                const int st = flow_ld(&sh.stop);
                on = !(st >= 0 && st <= known);
            }
            if (!__all_sync(0xffffffffu, on)) break;
            last = pass;
            // the impulses after pass s are in array s % 3
            const TP* Pin = (const TP*)flow_impulses(w, apply_only ? 0 : pass - 1);
            TP* Pout = (TP*)flow_impulses(w, pass);
            const bool save = pass >= FLOW_LAG1;
            T4* Vsave = Vprev + (size_t)(pass & 1) * RW * nprev;
            double acc = 0.0;
            bool owed = false;
            bool dead = false;
            int k = 0;
            auto settle = [&]() {   // the magnitude owed
                if constexpr (DEFER) {
                    if (owed) {
                        if constexpr (F64_2D) acc += abs_of_pair(pend.x, pend.y);
                        else if constexpr (DIM == 2) acc += abs_of_sq<T>((double)fma_of<T>(pend.y, pend.y, mul_of<T>(pend.x, pend.x)));
                        else acc += abs_of_sq<T>((double)fma_of<T>(pend.w, pend.w, fma_of<T>(pend.z, pend.z, fma_of<T>(pend.y, pend.y, mul_of<T>(pend.x, pend.x)))));
                    }
                    owed = false;
                }
            };
            for (int q = wid; q < Q; q += FLOW_WORKERS) {
                while (q >= sh.base[k + 1]) ++k;
                const int first = sh.lo[k], cnt = sh.end[k] - first;
                const bool split = F64_2D && sh.half[k];
                const int at = split ? 16 * (q - sh.base[k]) + (lane >> 1) : 32 * (q - sh.base[k]) + lane;
                const bool act = at < cnt;
                if constexpr (VIEWS) {
                    if (k == K) {
                        if (!flow_sum_views<DIM, T>(g, w, ctrl, sh, VT, vbase, first + at, act, pass)) { dead = true; break; }
                        if (gate) {
                            __syncwarp();
                            if (lane == 0) atomicAdd(&sh.done[k], 1);
                        }
                        continue;
                    }
                }
                const int p = first + at, i = sh.slot[k] + at;
                Rec<DIM, T> r;
                u64 *pa = nullptr, *pb = nullptr;
                unsigned ta = 0, tb = 0, ord = 0;
                bool wall = true;
                Body A, B;
                if (act) {
                    if (res) {
                        r.ab = rec.ab[i];   // (the records)
                        ord = rec.ord[i];
                    } else {
                        r.ab = VIEWS ? w.c_vab[p] : w.c_ab[p];
                        ord = w.fl_ord[p];
                    }
                    wall = !flow_moves<VIEWS>(g, r.ab.y);
                    ta = (unsigned)pass * ((ord >> 8) & 255u) + (ord & 255u);
                    tb = (unsigned)pass * (ord >> 24) + ((ord >> 16) & 255u);
                    pa = VT + (size_t)EB * r.ab.x;
                    if (!wall) pb = VT + (size_t)EB * r.ab.y;
                    if (!gate) {
                        A.load(pa);
                        if (!wall) B.load(pb);
                    }
                    // the rest of the record while the velocities are on their way
                    TM m;
                    if (res) {
                        const T2 t0 = rec.s0[i], t1 = rec.s1[i], t2 = rec.s2[i];
                        r.sa.x = t0.x; r.sa.y = t0.y; r.sa.z = t1.x; r.sa.w = (T)0;
                        r.sb.x = t1.y; r.sb.y = t2.x; r.sb.z = t2.y; r.sb.w = (T)0;
                        r.geo = rec.geo[i];
                        m = rec.m[i];
                        r.P = rec.P[i];
                    } else {
                        if constexpr (VIEWS) {
                            const int2 rr = r.ab;
                            r.ab = w.c_ab[p];
                            load_static<DIM, T>(g, w, r);
                            r.ab = rr;
                        } else {
                            load_static<DIM, T>(g, w, r);
                        }
                        r.geo = ((const T4*)w.c_geo)[p];
                        m = ((const TM*)w.c_m)[p];
                        r.P = Pin[p];
                    }
                    if constexpr (DIM == 2) r.mt = m;
                    else r.m = m;
                    r.pk = 0;
                    r.mu = mu;
                }
                // In a gas nearly every contact found is open and stays so (of a million
                // spheres' 912,728, one in 2,000 is not): an item whose contacts all are
                // takes the normal rate only, 23 of 79 FP64 instructions (2D: 6 of 25), and
                // nothing in the starting pass.  (Not where pairs of lanes share contacts: there
                // the votes in the chain cost more, 5,000 packed discs 19.9 -> 21.4 ms, than
                // a thin gas gains.)
                const bool shut = !split && __all_sync(0xffffffffu, !act || flow_zero(r.P));
                FlowHalf half;
                if constexpr (F64_2D) {
                    if (split) {
                        if (!act) {
                            r.geo.x = r.geo.y = r.geo.z = r.geo.w = 0.0;
                            r.sa = r.sb = r.geo;
                            r.P.x = r.P.y = r.mt = r.mu = 0.0;
                        }
                        half.choose(lane & 1, r);
                    }
                }
                if (gate) {
                    settle();
                    // not before the block's items of the colour before are done: the records are
                    // hardly there earlier, and looks that find nothing delay every other access
                    const int kb = sh.before[k] >= 0 ? sh.before[k] : -1 - sh.before[k];
                    const int need = (sh.base[kb + 1] - sh.base[kb]) * (pass + (sh.before[k] >= 0));
                    if (!__all_sync(0xffffffffu, flow_wait_shared(ctrl, sh, &sh.done[kb], need))) { dead = true; break; }
                    if (pa) A.load(pa);
                    if (pb) B.load(pb);
                }
                bool ra = !pa || A.has(ta), rb = !pb || B.has(tb);
                if (!__all_sync(0xffffffffu, ra && rb)) {
                    settle();   // in the wait, or else after this item's records are stored
                    if (!flow_wait<DIM, T>(ctrl, &sh.dead, pa, ta, pb, tb, A, B, ra, rb)) { dead = true; break; }
                }
                T4 va, oa, vb, ob;
                if constexpr (F64_2D) {
                    if (split) {
                        const bool odd = lane & 1;
                        if (act) {
                            A.unpack(va, oa);
                            if (!wall) B.unpack(vb, ob);
                            else wall_vel2<T>(g, w, r.ab.y, vb);
                        } else {
                            va.x = va.y = va.z = 0.0;
                            vb = va;
                        }
                        T4 v1;
                        const double Pnew = half.update(odd, r, va, vb, (wall || VIEWS) ? -1 : r.ab.y - g.n, apply_only, v1);
                        if (act && !(odd && wall)) {
                            A.pack(v1, v1, (odd ? tb : ta) + 1u);
                            A.store(odd ? pb : pa);
                        }
                        if (act) {
                            if (!apply_only) {
                                reinterpret_cast<double*>(Pout + p)[odd] = Pnew;
                                if (res) reinterpret_cast<double*>(rec.P + i)[odd] = Pnew;
                            }
                            // the records of the pass start, for taking the sweep back
                            const int mine = odd ? (int)((ord >> 16) & 255u) : (int)(ord & 255u);
                            const int body = odd ? r.ab.y : r.ab.x;
                            if (save && mine == 0 && !(odd && wall) && (!VIEWS || body < nprev)) Vsave[body] = odd ? vb : va;
                        }
                        settle();
                        const double Pother = shfl_pair(Pnew);
                        pend.x = Pnew;
                        pend.y = Pother;
                        owed = act && !odd;
                        __syncwarp();
                        if (gate && lane == 0) atomicAdd(&sh.done[k], 1);
                        continue;
                    }
                }
                if (act) {
                    A.unpack(va, oa);
                    if (!wall) B.unpack(vb, ob);
                    else if constexpr (DIM == 2) wall_vel2<T>(g, w, r.ab.y, vb);
                    else wall_vel3<T>(g, w, r.ab.y, vb, ob);
                }
                const bool still = shut && (apply_only || __all_sync(0xffffffffu, !act || flow_stays_open<T>(r, va, oa, vb, ob)));
                if (act) {
                    if (save) {
                        if ((ord & 255u) == 0u && (!VIEWS || r.ab.x < nprev)) {
                            Vsave[RW * r.ab.x] = va;
                            if constexpr (DIM == 3) Vsave[RW * r.ab.x + 1] = oa;
                        }
                        if (!wall && ((ord >> 16) & 255u) == 0u && (!VIEWS || r.ab.y < nprev)) {
                            Vsave[RW * r.ab.y] = vb;
                            if constexpr (DIM == 3) Vsave[RW * r.ab.y + 1] = ob;
                        }
                    }
                    TP Pn = r.P;
                    UpdOut o;
                    o.pabs = 0.0;
                    if (!still) {
                        if constexpr (DIM == 2) o = core2d<T, true>(g, r, va, vb, wall, apply_only, crit, alpha, 0.0, Pn);
                        else o = core3d<T, DEFER>(g, r, va, oa, vb, ob, wall, apply_only, crit, alpha, 0.0, Pn);
                    }
                    if (!VIEWS && !wall && r.ab.y >= g.n) {   // a force-controlled wall moves along its normal only
                        const int ax = (r.ab.y - g.n) >> 1;
                        if (ax != 0) vb.x = (T)0;
                        if (ax != 1) vb.y = (T)0;
                        if (DIM == 2 || ax != 2) vb.z = (T)0;
                        if constexpr (DIM == 3) ob.x = ob.y = ob.z = (T)0;
                    }
                    A.pack(va, oa, ta + 1u);
                    A.store(pa);
                    if (!wall) {
                        B.pack(vb, ob, tb + 1u);
                        B.store(pb);
                    }
                    if (!apply_only) {
                        Pout[p] = Pn;
                        if (res) rec.P[i] = Pn;
                    }
                    settle();
                    if constexpr (DEFER) {
                        pend = Pn;
                        owed = !still;
                    } else {
                        acc += o.pabs;
                    }
                }
                if (gate) {
                    __syncwarp();
                    if (lane == 0) atomicAdd(&sh.done[k], 1);
                }
            }
            if (dead) break;
            settle();
            *(volatile double*)&sh.acc[pass % FLOW_SLOTS][wid][lane] = acc;
            __syncwarp();
            if (lane == 0) {
                __threadfence_block();
                atomicAdd(&sh.arrived[pass % FLOW_SLOTS], 1);
            }
        }
    }
    __syncthreads();
    if (sh.dead) return false;
    const int sweeps = sh.stop;
    // final impulses of this block's contacts
    if (BATCH || sweeps % 3) {
        const TP* P = (const TP*)flow_impulses(w, sweeps);
        for (int k = 0; k < K; ++k)
            for (int p = sh.lo[k] + (int)threadIdx.x; p < sh.end[k]; p += blockDim.x) {
                const TP x = P[p];
                if constexpr (BATCH) {
                    const size_t c = (size_t)w.perm[p];
                    if constexpr (DIM == 2) {
                        w.Pk[2 * c] = (double)x.x; w.Pk[2 * c + 1] = (double)x.y;
                    } else {
                        w.Pk[4 * c] = (double)x.x; w.Pk[4 * c + 1] = (double)x.y;
                        w.Pk[4 * c + 2] = (double)x.z; w.Pk[4 * c + 3] = (double)x.w;
                    }
                } else {
                    ((TP*)w.c_P)[p] = x;
                }
            }
    }
    // sweeps past the last: the velocities from before them
    const bool back = __syncthreads_or(last > sweeps);
    if (!tm.sync(ctrl)) return false;
    for (int i = body0 + tid; i < body1; i += stride) {
        if (!cd_is_body(g, i)) continue;
        T4 v, o;
        if (back && w.fl_mask[i] != 0ULL) {
            const T4* Vsave = Vprev + (size_t)((sweeps + 1) & 1) * RW * nprev;
            v = Vsave[RW * i];
            v.w = (T)0;
            if constexpr (DIM == 3) o = Vsave[RW * i + 1];
        } else {
            Body x;
            x.load(VT + (size_t)EB * i);
            x.unpack(v, o);
        }
        V[RW * i] = v;
        if constexpr (DIM == 3) V[RW * i + 1] = o;
        if (!BATCH && io.vel && i < g.n) unpack_particle<DIM, T>(g, io, i, v, o);
    }
    return true;
}

// A plain system: the whole grid is one team.
template <int DIM, typename T, bool VIEWS>
__global__ void __launch_bounds__(FLOW_THREADS, 1)
k_flow(CdGeom g, CdWork w, CdState io, int crit, double alpha, int max_sweeps, int rec_cap)
{
    extern __shared__ __align__(128) char s_rec[];
    __shared__ FlowShared sh;
    __shared__ double s_red[FLOW_WORKERS + 1][3];
    CdCtrl* ctrl = w.ctrl;
    if (ctrl->skip) return;
    // (a set without contacts may have no colour order: a checkpoint can bring one)
    const int nc = ctrl->nc, K = nc > 0 ? ctrl->ncolours : 0, nb = gridDim.x;
    const FlowTeam tm{reinterpret_cast<unsigned*>(&ctrl->bar_count), 0, nb, (int)blockIdx.x, nb};
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        sh.lo[k] = w.colour_off[k];
        sh.end[k] = w.colour_off[k + 1];
    }
    __syncthreads();
    if (!flow_solve<DIM, T, false, VIEWS>(g, w, sh, s_rec, rec_cap, tm, io, K, nc, (T)g.mu, 0,
                                          g.n + (g.dyn_walls ? 6 : 0), crit, alpha, max_sweeps))
        return;
    u64 epoch = 0;
    finish_solve<DIM, T>(g, w, nc, nb, blockIdx.x * blockDim.x + threadIdx.x, nb * blockDim.x, epoch, sh.stop,
                         sh.converged, sh.resid, sh.ravg, s_red);
    if (io.vel && blockIdx.x == 0 && threadIdx.x == 0) {
        if (g.dyn_walls) unpack_walls<DIM, T>(g, w);   // (their records are written before the barrier in finish_solve)
        if (io.integrate) move_walls<DIM>(g, w, 0);
    }
}

// ---------------------------------------------------------------------------
// Batched systems.  Packings share nothing, so each is solved by a team of its
// own and stops by itself: no barrier and no residual pass over the others.  A
// packing asks for a block per `target` contacts and is spread over exactly as
// many, whichever team takes it: the magnitudes are added up lane by lane, so
// with another number of blocks the mean would end in other digits.  The largest
// packings' teams are laid out in advance until the grid is full; a team that is
// done takes the largest packing left that asks for no more blocks than it has.
// What is left of the team becomes one of its own if it is a third as many or
// more, or near the end (the first part so keeps at least as many blocks as any
// packing left asks for: none is left over); before that fewer stay, without
// contacts, since blocks once cut off do not come back together for a large
// packing.  One step from zero
// forces against the barrier schedule, which swept all packings together and
// summed each one's |P| in a single block: 8 packings 45.4 -> 12.6 ms, 23 57.6
// -> 17.5, 64 94 -> 55, 128 150 -> 91, 300 356 -> 229, 512 537 -> 394; from 64 on
// the FP64 pipe bounds it (128: 67 ms).  With the blocks left over given contacts
// too, which depends on timing: 102, 228 and 379 for the last three.  Cut always:
// 91, 352, 715; for a third or more to the end: 105, 233, 395; for a half: 106, 246, 407; for a
// whole: 109, 278, 469; from 3 rounds before the end 100, 230, 395, from 6 91, 231, 394 (200
// packings 162 -> 178).  A reserve of 32 contacts for every colour in
// place of 128 for all: the fourth step of 64 packings, whose most crowded disc
// has 29 contacts, 379 ms against 173 (285 with barriers).
// ---------------------------------------------------------------------------
__device__ __forceinline__ int flow_ask(const CdWork& w, int b, int target, int blocks)
{
    const int nc = w.pk_coff[b + 1] - w.pk_coff[b];
    const int ask = (nc + target - 1) / target;
    return ask < 1 ? 1 : (ask > blocks ? blocks : ask);
}

// Whether a batch is left to the barrier schedule: by what a sweep of all packings
// takes by either, in us.  By dataflow a block has one packing at a time, `rounds` of them
// one after another (packings that ask for several blocks in proportion), and of
// each a chain of its colours, whose latency the contacts of one colour in one
// block hardly fill.  Behind barriers all packings' contacts of a colour fill it
// together, but every colour is a barrier of the grid, the sums of the tests
// are a block's per packing, one after another, the largest of them alone at the
// end, and more contacts than L2 holds come from memory every sweep.  The terms were
// fitted to 370 batches of 3 to 5,000 equal packings (10 to 40,000 discs or spheres, 4
// to 25 colours, 2,000 to 13 million contacts in all): to 7 to 14% of the dataflow's times and 3 to
// 5% of the barriers', and the faster one is taken but in 13, where it is up to 20%
// (most 6%) faster.  A sweep, dataflow / barriers: 150 packings of 30 discs
// 9.1 / 29 us, 600 34 / 38, 5,000 259 / 132; FP64, 2,000 of 100 spheres with 7 contacts
// each 750 / 253, 200 of 2,000 859 / 444; 2,000 of 3,000 discs 1,014 / 1,189.  (A gas, whose
// contacts stay open, takes the dataflow less than that, but nothing tells beforehand.)
struct FlowCost {
    float round, colour, item;                      // dataflow: a round, a colour in it, 32 contacts of it in a block
    float sweep, phase, contact, packing, largest;  // barriers: a sweep, a colour, a contact and a packing a block,
    float far, near;                                // a contact of the largest packing, one a block beyond `near`
};
static FlowCost flow_cost(int dim, int precision)
{
    if (dim == 2)
        return precision == CD_FP64
                   ? FlowCost{0.55f, 1.11f, 0.222f, 6.0f, 3.35f, 0.0080f, 2.65f, 0.0006f, 0.0059f, 3000.0f}
                   : FlowCost{1.39f, 0.75f, 0.096f, 5.3f, 2.70f, 0.0034f, 2.76f, 0.0006f, 0.0067f, 9000.0f};
    return precision == CD_FP64
               ? FlowCost{0.0f, 2.99f, 0.510f, 4.5f, 4.57f, 0.0193f, 2.65f, 0.0006f, 0.0084f, 3000.0f}
               : FlowCost{0.59f, 0.78f, 0.233f, 3.3f, 2.87f, 0.0056f, 2.72f, 0.0006f, 0.0062f, 9000.0f};
}
// K colours in all, `own` a packing; the packings ask for `asks` blocks.
__device__ __forceinline__ bool flow_leaves_batch(const FlowCost& c, int K, float own, int nc, int largest, int asks,
                                                  int npk, int blocks)
{
    const float rounds = (float)((asks + blocks - 1) / blocks);
    const float items = fmaxf((float)nc / ((float)asks * own * 32.0f), 1.0f);
    const float flow = rounds * (c.round + own * (c.colour + c.item * items));
    const float each = (float)nc / (float)blocks;
    const float barriers = c.sweep + (float)K * c.phase + c.largest * (float)largest + c.contact * each +
                           c.far * fmaxf(each - c.near, 0.0f) + c.packing * (float)npk / (float)blocks;
    return barriers < flow;
}

__global__ void k_flow_plan(CdGeom g, CdWork w, int blocks, int records, FlowCost cost)
{
    __shared__ int s_at[FLOW_MAX_BLOCKS + 1];   // packings that ask for i blocks, then the next place of theirs
    __shared__ int s_largest;
    if (w.ctrl->skip) return;
    FlowPlan* plan = w.fl_plan;
    // all packings at once if the blocks' records can hold them so
    const int room = blocks > 2 * g.npk ? blocks - g.npk : blocks / 2;
    int target = (w.ctrl->nc + room - 1) / room;
    // (dealt in warp items, remainders from another block on for each colour, a block may get a few
    // more than its share; one that got too many would read them from memory)
    if (target > records - 128) target = records - 128;
    if (target < FLOW_LEAST) target = FLOW_LEAST;
    for (int i = threadIdx.x; i < 2 * g.npk + 1; i += blockDim.x) w.fl_word[i] = 0u;
    for (int i = threadIdx.x; i <= blocks; i += blockDim.x) s_at[i] = 0;
    if (threadIdx.x == 0) s_largest = 0;
    __syncthreads();
    for (int b = threadIdx.x; b < g.npk; b += blockDim.x) {
        atomicAdd(&s_at[flow_ask(w, b, target, blocks)], 1);
        atomicMax(&s_largest, w.pk_coff[b + 1] - w.pk_coff[b]);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        // the colours that a packing has of those there are: at most as many as there are contacts of
        // each for every packing, and one crowded packing's own weigh as much as their
        // contacts (1.25: in a packing alone the last colours have few)
        const int K = w.ctrl->ncolours, nc = w.ctrl->nc;
        float own = 0.0f, weight = 0.0f;
        for (int k = 0; k < K; ++k) {
            const float n = (float)(w.colour_off[k + 1] - w.colour_off[k]);
            own += fminf(1.0f, n / (float)g.npk);
            weight += fminf(1.0f, n * (float)K / (float)nc);
        }
        own = fmaxf(fminf(own, 1.25f * weight), 1.0f);
        int asks = 0;
        for (int ask = 1; ask <= blocks; ++ask) asks += ask * s_at[ask];
        plan->barriers = flow_leaves_batch(cost, K, own, nc, s_largest, asks, g.npk, blocks);
        int i = 0, run = 0, used = 0;
        bool full = false;
        for (int ask = blocks; ask >= 1; --ask) {
            const int n = s_at[ask];
            s_at[ask] = run;
            int placed = 0;   // of these
            while (placed < n && !full) {
                if (used + ask > blocks) { full = true; break; }
                w.fl_start[i++] = used;
                used += ask;
                ++placed;
            }
            plan->head[ask] = run + placed;
            run += n;
            plan->end[ask] = run;
        }
        w.fl_start[i] = used;
        plan->left = asks - used;
        plan->target = target;
        plan->placed = i;
    }
    __syncthreads();
    for (int b = threadIdx.x; b < g.npk; b += blockDim.x)
        w.fl_list[atomicAdd(&s_at[flow_ask(w, b, target, blocks)], 1)] = b;
}

// Takes the packing that asks for most blocks, but no more than nb: its place
// in fl_list, or -1 if none is left.  One warp.
__device__ __forceinline__ int flow_take(FlowPlan* plan, int nb)
{
    const int lane = threadIdx.x & 31;
    for (int g0 = nb; g0 >= 1; g0 -= 32) {
        const int ask = g0 - lane;
        const int end = ask >= 1 ? plan->end[ask] : 0;
        unsigned m = __ballot_sync(0xffffffffu, ask >= 1 && cd_ld_volatile_int(&plan->head[ask]) < end);
        while (m) {
            const int at = __ffs(m) - 1;
            int x = (lane == at) ? atomicAdd(&plan->head[ask], 1) : 0;
            if (lane == at && x >= end) x = -1;
            x = __shfl_sync(0xffffffffu, x, at);
            if (x >= 0) return x;
            m &= m - 1u;
        }
    }
    return -1;
}

// First position in [lo, hi) (one colour, key order) whose contact's body a is
// at least `particle`.
__device__ __forceinline__ int flow_lower(const CdWork& w, int lo, int hi, int particle)
{
    while (lo < hi) {
        const int mid = lo + ((hi - lo) >> 1);
        if (w.c_ab[mid].x < particle) lo = mid + 1; else hi = mid;
    }
    return lo;
}

template <int DIM, typename T>
__global__ void __launch_bounds__(FLOW_THREADS, 1)
k_flow_batch(CdGeom g, CdWork w, int crit, double alpha, int max_sweeps, int rec_cap)
{
    extern __shared__ __align__(128) char s_rec[];
    __shared__ FlowShared sh;
    __shared__ double s_red[FLOW_WORKERS + 1][3];
    CdCtrl* ctrl = w.ctrl;
    if (ctrl->skip || w.fl_plan->barriers) return;
    FlowPlan* plan = w.fl_plan;
    const int K = ctrl->ncolours, me = blockIdx.x, target = plan->target, placed = plan->placed;
    // the block's first team
    int at = 0, start = w.fl_start[placed], nb = (int)gridDim.x - start, slot = 2 * g.npk;
    bool given = me < start;
    if (given) {
        int hi = placed - 1;   // the last team that starts at or before this block
        while (at < hi) {
            const int mid = (at + hi + 1) >> 1;
            if (w.fl_start[mid] <= me) at = mid; else hi = mid - 1;
        }
        start = w.fl_start[at];
        nb = w.fl_start[at + 1] - start;
    }
    for (;;) {
        while (!given) {
            // the team of `slot` takes the next packing
            const FlowTeam tm{&w.fl_word[slot], start, nb, me - start, nb};
            if (tm.blk == 0 && threadIdx.x < 32) {
                const int x = flow_take(plan, nb);
                if (threadIdx.x == 0) {
                    int mail = -1;
                    if (x >= 0) {
                        // whether what is left over becomes a team of its own
                        const int ask = flow_ask(w, w.fl_list[x], target, (int)gridDim.x);
                        const int left = atomicSub(&plan->left, ask) - ask;
                        mail = 2 * x + (3 * nb >= 4 * ask || left < FLOW_TAIL * (int)gridDim.x ? 1 : 0);
                    }
                    *(volatile int*)&w.fl_mail[slot] = mail;
                }
            }
            if (!tm.sync(ctrl)) return;
            at = cd_ld_volatile_int(&w.fl_mail[slot]);
            if (at < 0) return;
            const bool cut = at & 1;
            at >>= 1;
            const int ask = flow_ask(w, w.fl_list[at], target, (int)gridDim.x);
            if (!cut || nb == ask) break;
            given = me < start + ask;
            if (given) {
                nb = ask;
            } else {
                start += ask;
                nb -= ask;
                slot = g.npk + at;
            }
        }
        given = false;
        slot = at;
        const int b = w.fl_list[at];
        const FlowTeam tm{&w.fl_word[slot], start, nb, me - start, flow_ask(w, b, target, (int)gridDim.x)};
        const int first = w.pk[b].first, count = w.pk[b].count;
        const int c0 = w.pk_coff[b], nc = w.pk_coff[b + 1] - c0;
        for (int k = threadIdx.x; k < K; k += blockDim.x) {
            const int lo = flow_lower(w, w.colour_off[k], w.colour_off[k + 1], first);
            sh.lo[k] = lo;
            sh.end[k] = flow_lower(w, lo, w.colour_off[k + 1], first + count);
        }
        __syncthreads();
        if (!flow_solve<DIM, T, true, false>(g, w, sh, s_rec, rec_cap, tm, CdState{nullptr, nullptr, nullptr, nullptr, 0}, K, nc, (T)w.pk[b].mu, first, first + count, crit,
                                      alpha, max_sweeps))
            return;
        if (tm.blk == 0) {
            // the packing's wall forces and statistics
            const int pw = (DIM == 2) ? 2 : 4;
            double lo3[3] = {0.0, 0.0, 0.0}, hi3[3] = {0.0, 0.0, 0.0};
            for (int i = c0 + (int)threadIdx.x; i < c0 + nc; i += blockDim.x) {
                const int bb = w.pairs[i].y;
                if (bb < g.n) continue;
                const int k = (bb - g.n) % 6;
                const double pn = w.Pk[pw * i];
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
                st[PKS_SWEEPS] = (double)sh.stop;
                st[PKS_CONV] = (double)sh.converged;
                st[PKS_RESID] = sh.resid;
                st[PKS_RAVG] = sh.ravg;
                st[PKS_RPREV] = sh.ravg;
                st[PKS_NC] = (double)nc;
                for (int q = 0; q < 3; ++q) {
                    st[PKS_WF0 + q] = lo3[q] / g.dt;
                    st[PKS_WF0 + 3 + q] = hi3[q] / g.dt;
                }
            }
        }
    }
}

// The call's totals over the packings.
__global__ void k_flow_totals(CdGeom g, CdWork w)
{
    __shared__ long long s_sum, s_upd, s_open;
    __shared__ int s_max;
    CdCtrl* ctrl = w.ctrl;
    if (ctrl->skip || ctrl->error != CDE_NONE || w.fl_plan->barriers) return;
    if (threadIdx.x == 0) { s_sum = 0; s_upd = 0; s_open = 0; s_max = 0; }
    __syncthreads();
    for (int b = threadIdx.x; b < g.npk; b += blockDim.x) {
        const double* st = w.pk_stats + CD_PKSTATS * b;
        const long long sw = (long long)st[PKS_SWEEPS];
        atomicAdd((unsigned long long*)&s_sum, (unsigned long long)sw);
        atomicAdd((unsigned long long*)&s_upd, (unsigned long long)(sw * (long long)st[PKS_NC]));
        if (st[PKS_CONV] == 0.0) atomicAdd((unsigned long long*)&s_open, 1ULL);
        atomicMax(&s_max, (int)sw);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const double* st = w.pk_stats;
        for (int q = 0; q < 6; ++q) ctrl->wall_force[q] = st[PKS_WF0 + q];
        ctrl->r_avg = st[PKS_RAVG];
        ctrl->residual = st[PKS_RESID];
        ctrl->steps_done += 1;
        ctrl->total_sweeps += s_sum;
        ctrl->total_updates += s_upd;
        ctrl->n_not_conv += s_open;
        if (s_max > ctrl->max_sweeps_step) ctrl->max_sweeps_step = s_max;
        ctrl->sweeps = s_max;
        ctrl->converged = (s_open == 0);
    }
}

enum { FLOW_PLAIN = 0, FLOW_BATCH, FLOW_VIEWS };
struct FlowKernel { const void* fn; int body_bytes, record_bytes; };
static FlowKernel flow_kernel(int dim, int precision, int kind)
{
#define FLOW_K(D, T) \
    FlowKernel{kind == FLOW_BATCH ? (const void*)k_flow_batch<D, T> \
               : kind == FLOW_VIEWS ? (const void*)k_flow<D, T, true> : (const void*)k_flow<D, T, false>, \
               (int)sizeof(FlowBody<D, T>), FlowRecords<D, T>::BYTES}
    if (dim == 2) return precision == CD_FP64 ? FLOW_K(2, double) : FLOW_K(2, float);
    return precision == CD_FP64 ? FLOW_K(3, double) : FLOW_K(3, float);
#undef FLOW_K
}

size_t cd_flow_body_bytes(int dim, int precision) { return (size_t)flow_kernel(dim, precision, FLOW_PLAIN).body_bytes; }

static int flow_kind(const CdGeom& g)
{
    return g.npk > 1 ? FLOW_BATCH : g.ndom_total > 1 ? FLOW_VIEWS : FLOW_PLAIN;
}

// Contacts a block keeps in shared memory (a multiple of 16, so that every
// array of the records stays aligned), or -1 if the kernel does not fit.
int cd_flow_records(const CdGeom& g, int precision, int device)
{
    const FlowKernel f = flow_kernel(g.dim, precision, flow_kind(g));
    int most = 0;
    cudaFuncAttributes a;
    if (cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) != cudaSuccess ||
        cudaFuncGetAttributes(&a, f.fn) != cudaSuccess)
        return -1;
    const int room = most - (int)a.sharedSizeBytes - 256;
    const int recs = room > 0 ? room / f.record_bytes / 16 * 16 : 0;
    if (cudaFuncSetAttribute(f.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, recs * f.record_bytes) != cudaSuccess)
        return -1;
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, f.fn, FLOW_THREADS, (size_t)(recs * f.record_bytes)) !=
            cudaSuccess || b < 1)
        return -1;
    return recs;
}

// Particles up to which the dataflow is the faster schedule.  A system whose
// contacts do not fit the blocks' shared memory is read through the L1, 11 warps an
// SM at a time; the barrier schedule has 16, each with its next record on the way,
// and barriers that weigh less the more there is between them.  A step of 150
// sweeps (FP32: also 2 to 3 of a gas), dataflow / barriers: FP32 packed discs
// 300,000 5.66 / 5.73 ms, 400,000 5.99 / 5.98, 700,000 11.4 / 8.1, 2,000,000 37.2 /
// 21.2, lattice of 16 contacts each 200,000 14.4 / 16.2, 400,000 28.1 / 25.9; FP32
// spheres, six contacts each, 150,000 5.00 / 5.23, 200,000 6.87 / 6.64, 400,000 13.3 /
// 9.5, 11 each 100,000 9.9 / 10.8, 200,000 16.8 / 14.7, a gas 400,000 0.58 / 0.55,
// 2,000,000 2.18 / 1.99; FP64 discs 700,000 17.6 / 19.3, 1,000,000 26.8 / 25.8,
// 2,000,000 57.1 / 49.5; FP64 spheres 2,000,000 124 / 132, a gas of 4,000,000
// 4.76 / 4.97: no line.  (With more contacts a body there are more colours, so as
// much to do in each: the line is one of particles.)
int64_t cd_flow_max_n(int dim, int precision, int blocks)
{
    if (precision == CD_FP32) return (int64_t)blocks * (dim == 2 ? 2300 : 1100);
    return dim == 2 ? (int64_t)blocks * 6000 : INT64_MAX;
}

static cudaError_t flow_launch(const CdGeom& g, const CdWork& w, const CdState* io, int blocks, int records, int precision, int criterion,
                               double alpha, int max_sweeps, cudaStream_t s, int* nl)
{
    cudaError_t e = cudaMemsetAsync(w.ctrl, 0, 2 * sizeof(u64), s);
    if (e != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(w.fl_mask, 0, sizeof(u64) * (size_t)w.fl_nrec, s)) != cudaSuccess) return e;
    const FlowKernel f = flow_kernel(g.dim, precision, flow_kind(g));
    CdGeom ga = g;
    CdWork wa = w;
    int crit = criterion, ms = max_sweeps, rc = records;
    double al = alpha;
    CdState st = io ? *io : CdState{nullptr, nullptr, nullptr, nullptr, 0};
    void* plain[] = {&ga, &wa, &st, &crit, &al, &ms, &rc};
    void* batch[] = {&ga, &wa, &crit, &al, &ms, &rc};
    ++*nl;
    return cudaLaunchCooperativeKernel(f.fn, dim3(blocks), dim3(FLOW_THREADS), io ? plain : batch,
                                       (size_t)(records * f.record_bytes), s);
}

cudaError_t cd_launch_flow(const CdGeom& g, const CdWork& w, const CdState& io, int blocks, int records, int precision, int criterion,
                           double alpha, int max_sweeps, cudaStream_t s, int* nl)
{
    return flow_launch(g, w, &io, blocks, records, precision, criterion, alpha, max_sweeps, s, nl);
}

cudaError_t cd_launch_flow_batch(const CdGeom& g, const CdWork& w, int blocks, int records, int precision,
                                 int criterion, double alpha, int max_sweeps, cudaStream_t s, int* nl)
{
    k_flow_plan<<<1, 512, 0, s>>>(g, w, blocks, records, flow_cost(g.dim, precision));
    ++*nl;
    cudaError_t e = flow_launch(g, w, nullptr, blocks, records, precision, criterion, alpha, max_sweeps, s, nl);
    if (e != cudaSuccess) return e;
    k_flow_totals<<<1, 256, 0, s>>>(g, w);
    ++*nl;
    return cudaGetLastError();
}
