// cd_sweep_core.cuh -- the single-contact update (paper Sec. 2.1, Fig. 2), its
// records and the deterministic reductions, shared by the sweep kernels.
#pragma once

#include <type_traits>

#include "cd_internal.cuh"

template <typename T> struct Vec;
// FP64 records are 32 bytes at 32-byte aligned addresses (every workspace array
// is 256-byte aligned): one 256-bit access per record
template <> struct Vec<double> { typedef double4_32a V4; typedef double2 V2; };
template <> struct Vec<float> { typedef float4 V4; typedef float2 V2; };

// Arithmetic of the sweep's real type with the rounding written out (no
// contraction left to the compiler): fused multiply-add rounded once,
// product, sum and difference.
template <typename T> __device__ __forceinline__ T fma_of(T a, T b, T c);
template <> __device__ __forceinline__ double fma_of<double>(double a, double b, double c) { return __fma_rn(a, b, c); }
template <> __device__ __forceinline__ float fma_of<float>(float a, float b, float c) { return __fmaf_rn(a, b, c); }
template <typename T> __device__ __forceinline__ T mul_of(T a, T b);
template <> __device__ __forceinline__ double mul_of<double>(double a, double b) { return __dmul_rn(a, b); }
template <> __device__ __forceinline__ float mul_of<float>(float a, float b) { return __fmul_rn(a, b); }
template <typename T> __device__ __forceinline__ T add_of(T a, T b);
template <> __device__ __forceinline__ double add_of<double>(double a, double b) { return __dadd_rn(a, b); }
template <> __device__ __forceinline__ float add_of<float>(float a, float b) { return __fadd_rn(a, b); }
template <typename T> __device__ __forceinline__ T sub_of(T a, T b);
template <> __device__ __forceinline__ double sub_of<double>(double a, double b) { return __dsub_rn(a, b); }
template <> __device__ __forceinline__ float sub_of<float>(float a, float b) { return __fsub_rn(a, b); }

// Stores the first three components of a velocity record, leaving the fourth.
template <typename T>
__device__ __forceinline__ void store_xyz_plain(typename Vec<T>::V4* dst, const typename Vec<T>::V4& v)
{
    typedef typename Vec<T>::V2 T2;
    T2 xy;
    xy.x = v.x; xy.y = v.y;
    *reinterpret_cast<T2*>(dst) = xy;
    reinterpret_cast<T*>(dst)[2] = v.z;
}

// ---------------------------------------------------------------------------
// Deterministic reductions
// ---------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sum over the warp, or +0 without any FP64 instruction when every lane
// holds +0 (a warp of idle threads: the narrow FP64 pipe would spend the
// same time on it as on a busy warp).  The same bits as warp_sum.
__device__ __forceinline__ double warp_sum_nz(double v)
{
    if (!__any_sync(0xffffffffu, __double_as_longlong(v) != 0)) return v;
    return warp_sum(v);
}

// Block sum of the first nv of NV values per thread (fixed tree); result
// valid in thread 0.  Values nv .. NV-1 stay the thread's own (callers pass
// nv < NV only when those values are zero everywhere).
template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV], double (*s_red)[NV], int nv = NV)
{
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int j = 0; j < NV; ++j)
        if (j < nv) v[j] = warp_sum_nz(v[j]);
    if (lane == 0)
#pragma unroll
        for (int j = 0; j < NV; ++j)
            if (j < nv) s_red[wid][j] = v[j];
    __syncthreads();
    if (wid == 0) {
        int nw = blockDim.x >> 5;
#pragma unroll
        for (int j = 0; j < NV; ++j) {
            if (j < nv) {
                double x = (lane < nw) ? s_red[lane][j] : 0.0;
                v[j] = warp_sum_nz(x);
            }
        }
    }
    __syncthreads();
}

// Sum over blocks of partial field f, identical in every block: lanes of warp
// 0 stride over the blocks in order, then a fixed butterfly; broadcast.
__device__ __forceinline__ double grid_total(const double* part, int nblocks, double* s_bcast)
{
    if (threadIdx.x < 32) {
        double x = 0.0;
        for (int b = threadIdx.x; b < nblocks; b += 32) x += part[b];
        x = warp_sum(x);
        if (threadIdx.x == 0) *s_bcast = x;
    }
    __syncthreads();
    double r = *s_bcast;
    __syncthreads();
    return r;
}

// Values of the per-block partials a sweep's convergence test reads (the
// counts of test II only under that test).
__device__ __forceinline__ int test_values(int crit) { return crit == CD_CONV_LOCAL ? 3 : 1; }

// The global convergence tests (the plain ratio, its square II, none) on the
// mean impulses ra of this sweep and ravg_prev of the one before; 0 / 0
// passes, a NaN never does.
__device__ __forceinline__ void global_test(double ra, double ravg_prev, int crit, double alpha, double& rs, int& cv)
{
    const double den = ra + ravg_prev;
    if (crit == CD_CONV_GLOBAL_SQ) {
        const double q = (den > 0.0) ? (ra - ravg_prev) / den : (den == 0.0 ? 0.0 : den);
        rs = q * q;
    } else {
        rs = (den > 0.0) ? fabs(ra - ravg_prev) / den : (den == 0.0 ? 0.0 : den);
    }
    cv = crit != CD_CONV_NONE && rs < alpha;
}

// The convergence test after a sweep (tests I and II) from the block
// partials part[0 .. 3 nb): the block's last warp sums them (the order of
// grid_total) and its lane 0 decides; the result reaches the block through
// shared memory (s_b3, three doubles), so the FP64 divisions run once per
// block.  The last warp holds the fewest contacts of a colour phase (they
// are dealt from thread 0 up), so the other warps' work before the block
// barrier below (the next sweep's first updates, staged) overlaps the test.
__device__ __forceinline__ void sweep_test(const double* part, int nb, int nc, int crit, double alpha,
                                           double ravg_prev, double& ravg, double& resid, int& converged,
                                           double* s_b3)
{
    if ((threadIdx.x >> 5) == (blockDim.x >> 5) - 1) {
        const int lane = threadIdx.x & 31;
        const bool local = (crit == CD_CONV_LOCAL);
        double x = 0.0, xr = 0.0, xb = 0.0;
        for (int b = lane; b < nb; b += 32) {
            x += part[b];
            if (local) { xr += part[nb + b]; xb += part[2 * nb + b]; }
        }
        x = warp_sum(x);
        if (local) { xr = warp_sum(xr); xb = warp_sum(xb); }
        if (lane == 0) {
            const double ra = x / (double)nc;
            double rs;
            int cv;
            if (local) {
                rs = (double)(nc - (long long)xr) / (double)nc;
                cv = (10.0 * xr >= 9.0 * (double)nc) && xb == 0.0;
            } else {
                global_test(ra, ravg_prev, crit, alpha, rs, cv);
            }
            s_b3[0] = ra;
            s_b3[1] = rs;
            s_b3[2] = (double)cv;
        }
    }
    __syncthreads();
    ravg = s_b3[0];
    resid = s_b3[1];
    converged = (s_b3[2] != 0.0);
    __syncthreads();
}

// ---------------------------------------------------------------------------
// Single-contact updates (Fig. 2).  A contact record holds everything of the
// update except the two bodies' velocities: it is read-only within a colour
// phase, so a thread loads its next record before the grid barrier and only
// the velocity loads sit on the critical path after it.
// ---------------------------------------------------------------------------
struct UpdOut {
    double pabs;     // |P| after the update (deferred form: |P| of the thread's previous update)
    double psq;      // |P|^2 after the update (3D and FP32)
    double pn, pt;   // deferred form (FP64 2D): P_n, P_t after the update
    int rel_ok;      // local test (I), relative branch
    int bad;         // local test (I): fails both branches
};

template <int DIM, typename T> struct Rec;
template <typename T> struct Rec<2, T> {
    typedef typename Vec<T>::V4 T4;
    typedef typename Vec<T>::V2 T2;
    T mu;        // friction coefficient of the contact's packing
    int pk;      // packing of body a
    int2 ab;
    T4 geo;      // nx, ny, b = g/dt, m_n
    T mt;
    T2 P;        // P_n, P_t before the update
    T4 sa, sb;   // inv_m, r, r/I, 0 (sb = 0 for a wall)
    int2 vab;    // domain-wise update only: velocity records of a and b
};
template <typename T> struct Rec<3, T> {
    typedef typename Vec<T>::V4 T4;
    typedef typename Vec<T>::V2 T2;
    T mu;
    int pk;
    int2 ab;
    T4 geo;      // nx, ny, nz, b = g/dt
    T2 m;        // m_n, m_t
    T4 P;        // P_n, P_tx, P_ty, P_tz before the update
    T4 sa, sb;
    int2 vab;
};

// The bodies' static records (inv_m, r, r/I).  FP64: loaded with the
// velocities, after the barrier, not with the prefetched record (their
// loads run in parallel with the velocity loads, and the record held across
// the barrier stays 16 registers smaller: no spills at the 128-register
// cap; 2D sweep 28.56 -> 28.28 ms per step).  FP32 (no spills, 16-byte
// records): with the prefetched record, which was 2% faster there.
template <int DIM, typename T>
__device__ __forceinline__ void load_static(const CdGeom& g, const CdWork& w, Rec<DIM, T>& r)
{
    typedef typename Vec<T>::V4 T4;
    const T4* S = (const T4*)w.S;
    r.sa = S[r.ab.x];
    if (cd_is_body(g, r.ab.y)) {   // a particle, or a force-controlled wall (record n + k)
        r.sb = S[r.ab.y];
    } else {
        r.sb.x = (T)0; r.sb.y = (T)0; r.sb.z = (T)0; r.sb.w = (T)0;
    }
}

// VIEWS: the domain-wise update, whose contacts work on their domain's
// velocity records (c_vab); otherwise the records are the bodies' own.
template <int DIM, typename T, bool VIEWS = false>
__device__ __forceinline__ void load_rec(const CdGeom& g, const CdWork& w, int pos, Rec<DIM, T>& r)
{
    typedef typename Vec<T>::V4 T4;
    typedef typename Vec<T>::V2 T2;
    r.ab = w.c_ab[pos];
    if (g.npk > 1) {
        r.pk = w.pack_of[r.ab.x];
        r.mu = (T)w.pk[r.pk].mu;
    } else {
        r.pk = 0;
        r.mu = (T)g.mu;
    }
    r.geo = ((const T4*)w.c_geo)[pos];
    if constexpr (DIM == 2) {
        r.mt = ((const T*)w.c_m)[pos];
        r.P = ((const T2*)w.c_P)[pos];
    } else {
        r.m = ((const T2*)w.c_m)[pos];
        r.P = ((const T4*)w.c_P)[pos];
    }
    if constexpr (sizeof(T) == 4) load_static<DIM, T>(g, w, r);
    if constexpr (VIEWS) r.vab = w.c_vab[pos];
}



// max(x, 0) and the projection of x onto [-lim, lim] (lim >= 0).  For FP64
// they are done on the bit patterns with integer instructions (non-negative
// doubles order like their 64-bit integer images), which keeps them off the
// narrow FP64 pipe; the results are exactly those of the comparisons.
__device__ __forceinline__ double pos_part(double x)
{
    long long b = __double_as_longlong(x);
    return b < 0 ? 0.0 : x;
}
__device__ __forceinline__ float pos_part(float x) { return x > 0.0f ? x : 0.0f; }

__device__ __forceinline__ double clamp_sym(double x, double lim)
{
    unsigned long long bx = (unsigned long long)__double_as_longlong(x);
    unsigned long long bl = (unsigned long long)__double_as_longlong(lim);
    unsigned long long ax = bx & 0x7FFFFFFFFFFFFFFFULL;
    return ax > bl ? __longlong_as_double((long long)(bl | (bx & 0x8000000000000000ULL))) : x;
}
__device__ __forceinline__ float clamp_sym(float x, float lim) { return x < -lim ? -lim : (x > lim ? lim : x); }

// |P| = sqrt(s) from |P|^2 for the residual only, in two FP64 instructions
// (the FP64 pipe is the narrow one).  Write s = m 4^k with m in [1, 4) by
// exponent arithmetic on the bit pattern; take the FP32 reciprocal square
// root z of m rounded to FP32 (correctly rounded, __frsqrt_rn) and the FP32
// product y = m z, both on the wide FP32 pipe and widened exactly; then one
// Newton step of Heron's iteration for sqrt(m) from y, with z / 2 for
// 1 / (2 y): y + (m - y^2) z / 2; scale by 2^k.  With y = sqrt(m) (1 + d),
// |d| <= 2.5 2^-24 (three FP32 roundings), and z sqrt(m) = 1 + e, |e| <=
// 1.5 2^-24, the result is sqrt(m) (1 - d^2 / 2 - d e + O(d^3)): within
// 2.5e-14 relative.  Subnormal and infinite s take
// s * rsqrt(s); zero and negative s give 0; a NaN with the sign bit clear
// (what arithmetic on NaN produces here) gives NaN, as sqrt would, so that a
// diverged iteration does not look converged to the residual test; the
// decision is on the bit pattern, with no FP64 compare.
__device__ __forceinline__ double norm_of_sq(double s)
{
    const long long b = __double_as_longlong(s);
    const int be = (int)(b >> 52);   // biased exponent (sign clear for s >= 0)
    if (be <= 0 || be >= 0x7FF)
        return (b > 0 && b <= 0x7FF0000000000000LL) ? s * rsqrt(s) : (b > 0x7FF0000000000000LL ? s : 0.0);
    const int e = be - 1023;
    const int k = e >> 1;   // floor(e / 2)
    const long long mb = (b & 0x000FFFFFFFFFFFFFLL) | ((long long)(1023 + e - 2 * k) << 52);
    const double m = __longlong_as_double(mb);
    // m to FP32, rounded to nearest (a carry into the exponent is the rounding)
    const float mf = __int_as_float((int)(((mb + (1LL << 28)) >> 29) - (896LL << 23)));
    const float zf = __frsqrt_rn(mf);   // in [0.5, 1]
    const long long zb = ((long long)__float_as_int(zf) << 29) + (896LL << 52);   // exact widening
    const double h = __longlong_as_double(zb - (1LL << 52));                      // z / 2
    const float yf = __fmul_rn(mf, zf);                                            // ~sqrt(m), in (0.9, 2.1)
    const double y = __longlong_as_double(((long long)__float_as_int(yf) << 29) + (896LL << 52));   // exact
    const double r = __fma_rn(-y, y, m);
    const double y1 = __fma_rn(r, h, y);
    return __longlong_as_double(__double_as_longlong(y1) + ((long long)k << 52));
}

// |P| from the |P|^2 an update left (in the sweep's real type: FP32 impulses
// carry 1e-7 anyway, their magnitude is taken in FP32).  The persistent FP64
// 2D sweep defers it: a thread takes the magnitude of its previous update
// while the velocity loads of its next one are in flight, when the narrow
// FP64 pipe has nothing else to do; the per-thread sum sees the same terms in
// the same order, so the residual is bit-identical.
template <typename T> __device__ __forceinline__ double abs_of_sq(double s);
template <> __device__ __forceinline__ double abs_of_sq<double>(double s) { return norm_of_sq(s); }
template <> __device__ __forceinline__ double abs_of_sq<float>(double s) { return (double)sqrtf((float)s); }

// |P|^2 = P_n^2 + P_t^2 with a fixed rounding (the FP64 2D sweeps take it
// either inline or deferred, and must agree), and |P| from the pair.
__device__ __forceinline__ double sq2(double a, double b) { return __fma_rn(b, b, __dmul_rn(a, a)); }

// |P| of a 2D impulse without an FP64 instruction: the squares as 64-bit
// integers, FP32 for the root, and its remainder against the exact square of
// that in integers again.  With the larger component scaled to [2^63, 2^64) and
// the other aligned to it, S = (X^2 + Z^2) / 2^65 is exact to 2^-60; y is the
// FP32 root of S's top bits (24 bits, relative error below 2^-23), S - y^2 is an
// integer of at most 42 bits, and y + (S - y^2) / (2 y) is the root to y's
// error squared.  The quotient is taken in FP32 with one remainder step and
// added to y's bit pattern.  Against the Newton step on the FP64 pipe above,
// over 4e6 pairs (exponents e^-10 to e^10; open, sticking, sliding): largest
// relative error 7.3e-15 (9.8e-15), rms 9.1e-16 (2.0e-15), mean 1.8e-16
// (-1.2e-15).  The FP64 pipe keeps one instruction of five a contact, the sum.
__device__ __forceinline__ double abs_of_pair(double pn, double pt)
{
    typedef unsigned long long u64;
    const u64 ua = (u64)__double_as_longlong(pn) & 0x7FFFFFFFFFFFFFFFULL;
    const u64 ub = (u64)__double_as_longlong(pt) & 0x7FFFFFFFFFFFFFFFULL;
    if ((ua | ub) == 0ULL) return 0.0;
    const int ea = (int)(ua >> 52), eb = (int)(ub >> 52), em = max(ea, eb);
    if (em < 64 || em > 1980) return norm_of_sq(sq2(pn, pt));   // near the ends of the range, infinite, NaN
    const u64 ma = ea ? (ua << 11) | (1ULL << 63) : 0ULL, mb = eb ? (ub << 11) | (1ULL << 63) : 0ULL;
    const int da = em - ea, db = em - eb;
    const u64 X = da > 63 ? 0ULL : ma >> da, Z = db > 63 ? 0ULL : mb >> db;
    const unsigned xh = (unsigned)(X >> 32), xl = (unsigned)X, zh = (unsigned)(Z >> 32), zl = (unsigned)Z;
    const u64 H = (u64)xh * xh + (((u64)xh * xl) >> 31), I = (u64)zh * zh + (((u64)zh * zl) >> 31);
    const u64 S = (H >> 1) + (I >> 1);   // |P|^2 2^61 with the larger component in [1, 2)
    const float y = __fsqrt_rn(__fmul_rn(__uint2float_rn((unsigned)(S >> 32)), 1.86264515e-9f));   // 2^-29
    const unsigned yb = (unsigned)__float_as_int(y);
    const int ey = (int)(yb >> 23) - 127;   // 0 or 1
    const unsigned ym = (yb & 0x7FFFFFu) | 0x800000u;
    const long long R = (long long)(S - (((u64)ym * ym) << (15 + 2 * ey)));
    // (S - y^2) / (2 y) in units of the last place of y as a double
    const float rf = __int2float_rn((int)(R >> 12));
    const float sc = ey ? 2.0f : 4.0f;
    const float rz = __fmul_rn(__frcp_rn(y), sc);
    const float q = __fmul_rn(rf, rz);
    const float q2 = __fmul_rn(__fmaf_rn(-q, __fmul_rn(y, ey ? 0.5f : 0.25f), rf), rz);
    const u64 Y = ((u64)yb << 29) + (896ULL << 52);
    const u64 r = Y + (u64)(long long)__float2int_rn(q) + (u64)(long long)__float2int_rn(q2);
    if ((r ^ Y) >> 52) return norm_of_sq(sq2(pn, pt));   // past a power of two: its last place is another
    return __longlong_as_double((long long)(r + ((u64)(long long)(em - 1023) << 52)));
}

// 2D: b + u_n.  (b in the first fused step would save an instruction, but a
// contact that carries rounding noise only, under a lid that hangs free for
// one, is then open where it was closed, and counts of contacts change.)
template <typename T>
__device__ __forceinline__ T gap_rate2d(T nx, T ny, T b, T dvx, T dvy)
{
    return add_of<T>(b, fma_of<T>(dvy, ny, mul_of<T>(dvx, nx)));
}

// Biased exponent of x, and whether x y is finite by those of the two with room
// for a few sums.
__device__ __forceinline__ int exponent_of(double x) { return (int)(__double_as_longlong(x) >> 52) & 0x7ff; }
__device__ __forceinline__ int exponent_of(float x) { return (__float_as_int(x) >> 23) & 0xff; }
template <typename T>
__device__ __forceinline__ bool tame(int ex, int ey)
{
    constexpr int top = sizeof(T) == 8 ? 0x7ff : 0xff;
    return max(ex, ey) < top - 8 && ex + ey < top / 2 + top - 8;
}

// A contact that was open (P = 0) stays so: its new normal impulse is 0, by the
// operations of the update.  (Where something is infinite or undefined, or
// might be in the tangential part, the update itself has to tell.)
template <typename T>
__device__ __forceinline__ bool stays_open(T mn, T bun)
{
    const T Pn = pos_part(fma_of<T>(-mn, bun, (T)0));
    if constexpr (sizeof(T) == 8) return exponent_of(bun) != 0x7ff && __double_as_longlong(Pn) == 0LL;   // (off the FP64 pipe)
    else return exponent_of(bun) != 0xff && Pn == (T)0;
}

// 2D: P_n = max(0, P_n,old - m_n (b + u_n)); P_t = clamp(P_t,old - m_t u_t, +-mu P_n).
template <typename T, bool SQ = false>
__device__ __forceinline__ UpdOut core2d(const CdGeom& g, const Rec<2, T>& r, typename Vec<T>::V4& va,
                                         typename Vec<T>::V4& vb, bool wall, bool apply_only, int crit,
                                         double alpha, double ravg_prev, typename Vec<T>::V2& Pnew)
{
    // every operation is written out (fused steps where they save an
    // instruction): each kernel and call site that inlines this computes the
    // same bits
    const T nx = r.geo.x, ny = r.geo.y;
    T Pn, Pt, dPn, dPt;
    if (apply_only) {
        Pn = r.P.x; Pt = r.P.y;
        dPn = Pn; dPt = Pt;
    } else {
        const T b = r.geo.z, mn = r.geo.w;
        const T dvx = sub_of<T>(vb.x, va.x), dvy = sub_of<T>(vb.y, va.y);
        const T bun = gap_rate2d<T>(nx, ny, b, dvx, dvy);
        // u_t = (dv x n) - (r_a w_a + r_b w_b)
        T ut = fma_of<T>(dvy, nx, -mul_of<T>(dvx, ny));
        ut = fma_of<T>(-r.sa.y, va.z, ut);
        ut = fma_of<T>(-r.sb.y, vb.z, ut);
        Pn = pos_part(fma_of<T>(-mn, bun, r.P.x));
        const T lim = mul_of<T>(r.mu, Pn);
        Pt = clamp_sym(fma_of<T>(-r.mt, ut, r.P.y), lim);
        dPn = sub_of<T>(Pn, r.P.x);
        dPt = sub_of<T>(Pt, r.P.y);
    }
    const T dPx = fma_of<T>(dPn, nx, -mul_of<T>(dPt, ny));
    const T dPy = fma_of<T>(dPn, ny, mul_of<T>(dPt, nx));
    va.x = fma_of<T>(-r.sa.x, dPx, va.x);
    va.y = fma_of<T>(-r.sa.x, dPy, va.y);
    va.z = fma_of<T>(-r.sa.z, dPt, va.z);
    if (!wall) {
        vb.x = fma_of<T>(r.sb.x, dPx, vb.x);
        vb.y = fma_of<T>(r.sb.x, dPy, vb.y);
        vb.z = fma_of<T>(-r.sb.z, dPt, vb.z);
    }
    Pnew.x = Pn; Pnew.y = Pt;
    UpdOut o;
    const double pn = (double)Pn, pt = (double)Pt;
    // SQ (FP64): the pair only, the magnitude is taken later (abs_of_pair)
    o.pn = pn;
    o.pt = pt;
    if constexpr (sizeof(T) == 4) {
        o.psq = (double)fma_of<T>(Pt, Pt, mul_of<T>(Pn, Pn));
        o.pabs = abs_of_sq<T>(o.psq);
    } else {
        o.psq = 0.0;
        o.pabs = SQ ? 0.0 : abs_of_pair(pn, pt);
    }
    o.rel_ok = 0; o.bad = 0;
    if (!apply_only && crit == CD_CONV_LOCAL) {
        const double d0 = (double)dPn, d1 = (double)dPt;
        const double s0 = __dadd_rn(pn, (double)r.P.x), s1 = __dadd_rn(pt, (double)r.P.y);
        const double d2 = sq2(d0, d1), s2 = sq2(s0, s1);
        o.rel_ok = d2 < __dmul_rn(alpha, s2);
        o.bad = !o.rel_ok && !(d2 <= __dmul_rn(__dmul_rn(alpha, ravg_prev), ravg_prev));
    }
    return o;
}

// Velocity of wall body n + 6 * packing + k.
__device__ __forceinline__ const double* wall_velocity(const CdGeom& g, const CdWork& w, int wid)
{
    const int t = wid - g.n;
    return (g.npk > 1) ? w.pk[t / 6].wall_vel + 3 * (t % 6) : g.wall_vel + 3 * t;
}

template <typename T>
__device__ __forceinline__ void wall_vel2(const CdGeom& g, const CdWork& w, int wid, typename Vec<T>::V4& vb)
{
    const double* u = wall_velocity(g, w, wid);
    vb.x = (T)u[0]; vb.y = (T)u[1]; vb.z = (T)0; vb.w = (T)0;
}

// VIEWS: the bodies' velocity records are the domain views r.vab, else their own.
// DEFER (FP64): the result's pabs is |P| of the thread's previous update,
// taken from its (P_n, P_t) `pend` after this update's velocity loads are
// issued; pn, pt hold this update's impulse.
// A 2D update computed but not yet stored: the two velocity records and the
// impulse, where they go.
template <typename T>
struct Staged2 {
    typename Vec<T>::V4 va, vb;
    typename Vec<T>::V2 P;
    int ia, ib, pos;
    bool wall, store_p;
};

template <typename T, bool VIEWS = false, bool DEFER = false>
__device__ __forceinline__ UpdOut stage2d(const CdGeom& g, const CdWork& w, int pos, const Rec<2, T>& r,
                                          bool apply_only, int crit, double alpha, double ravg_prev, double2 pend,
                                          Staged2<T>& st)
{
    typedef typename Vec<T>::V4 T4;
    const T4* V = (const T4*)w.V;
    st.ia = VIEWS ? r.vab.x : r.ab.x;
    st.ib = VIEWS ? r.vab.y : r.ab.y;
    st.pos = pos;
    st.store_p = !apply_only;
    st.wall = !cd_is_body(g, r.ab.y);   // kinematic wall
    st.va = V[st.ia];
    if (!st.wall) st.vb = V[st.ib];
    else wall_vel2<T>(g, w, r.ab.y, st.vb);
    Rec<2, T> rs = r;
    if constexpr (sizeof(T) == 8) load_static<2, T>(g, w, rs);
    const double prev = DEFER ? abs_of_pair(pend.x, pend.y) : 0.0;
    UpdOut o = core2d<T, DEFER>(g, rs, st.va, st.vb, st.wall, apply_only, crit, alpha, ravg_prev, st.P);
    if constexpr (DEFER) o.pabs = prev;
    if (!st.wall && r.ab.y >= g.n) {
        // a force-controlled wall moves along its normal only
        if (((r.ab.y - g.n) >> 1) == 0) st.vb.y = (T)0; else st.vb.x = (T)0;
        st.vb.z = (T)0;
    }
    return o;
}

template <typename T>
__device__ __forceinline__ void commit2d(const CdWork& w, const Staged2<T>& st)
{
    typedef typename Vec<T>::V4 T4;
    typedef typename Vec<T>::V2 T2;
    T4* V = (T4*)w.V;
    V[st.ia] = st.va;
    if (!st.wall) V[st.ib] = st.vb;
    if (st.store_p) ((T2*)w.c_P)[st.pos] = st.P;
}

template <typename T, bool VIEWS = false, bool DEFER = false>
__device__ __forceinline__ UpdOut apply2d(const CdGeom& g, const CdWork& w, int pos, const Rec<2, T>& r,
                                          bool apply_only, int crit, double alpha, double ravg_prev,
                                          double2 pend = make_double2(0.0, 0.0))
{
    Staged2<T> st;
    const UpdOut o = stage2d<T, VIEWS, DEFER>(g, w, pos, r, apply_only, crit, alpha, ravg_prev, pend, st);
    commit2d<T>(w, st);
    return o;
}

// 3D: relative velocity of the contact points, (vb - va) - (ra wa + rb wb) x n;
// returns its normal part.
template <typename T>
__device__ __forceinline__ T contact_velocity3d(const Rec<3, T>& r, const typename Vec<T>::V4& va,
                                                const typename Vec<T>::V4& wa, const typename Vec<T>::V4& vb,
                                                const typename Vec<T>::V4& wb, T& gx, T& gy, T& gz)
{
    const T nx = r.geo.x, ny = r.geo.y, nz = r.geo.z;
    const T lx = fma_of<T>(r.sb.y, wb.x, mul_of<T>(r.sa.y, wa.x));
    const T ly = fma_of<T>(r.sb.y, wb.y, mul_of<T>(r.sa.y, wa.y));
    const T lz = fma_of<T>(r.sb.y, wb.z, mul_of<T>(r.sa.y, wa.z));
    gx = sub_of<T>(sub_of<T>(vb.x, va.x), fma_of<T>(ly, nz, -mul_of<T>(lz, ny)));
    gy = sub_of<T>(sub_of<T>(vb.y, va.y), fma_of<T>(lz, nx, -mul_of<T>(lx, nz)));
    gz = sub_of<T>(sub_of<T>(vb.z, va.z), fma_of<T>(lx, ny, -mul_of<T>(ly, nx)));
    return fma_of<T>(gz, nz, fma_of<T>(gy, ny, mul_of<T>(gx, nx)));
}

// 3D: the same with the tangential impulse a vector, scaled onto the cone.
template <typename T, bool SQ = false>
__device__ __forceinline__ UpdOut core3d(const CdGeom& g, const Rec<3, T>& r, typename Vec<T>::V4& va,
                                         typename Vec<T>::V4& wa, typename Vec<T>::V4& vb, typename Vec<T>::V4& wb,
                                         bool wall, bool apply_only, int crit, double alpha, double ravg_prev,
                                         typename Vec<T>::V4& Pnew)
{
    // every operation written out, as in core2d
    const T nx = r.geo.x, ny = r.geo.y, nz = r.geo.z;
    T Pn, Ptx, Pty, Ptz, dPn, dtx, dty, dtz;
    if (apply_only) {
        Pn = r.P.x; Ptx = r.P.y; Pty = r.P.z; Ptz = r.P.w;
        dPn = Pn; dtx = Ptx; dty = Pty; dtz = Ptz;
    } else {
        const T mn = r.m.x, mt = r.m.y, b = r.geo.w;
        T gx, gy, gz;
        const T un = contact_velocity3d<T>(r, va, wa, vb, wb, gx, gy, gz);
        const T tx = fma_of<T>(-un, nx, gx), ty = fma_of<T>(-un, ny, gy), tz = fma_of<T>(-un, nz, gz);
        Pn = pos_part(fma_of<T>(-mn, add_of<T>(b, un), r.P.x));
        Ptx = fma_of<T>(-mt, tx, r.P.y);
        Pty = fma_of<T>(-mt, ty, r.P.z);
        Ptz = fma_of<T>(-mt, tz, r.P.w);
        const T lim = mul_of<T>(r.mu, Pn);
        const T q2 = fma_of<T>(Ptz, Ptz, fma_of<T>(Pty, Pty, mul_of<T>(Ptx, Ptx)));
        if (q2 > mul_of<T>(lim, lim)) {
            const T sc = mul_of<T>(lim, rsqrt(q2));   // onto the cone (q2 > lim^2 >= 0)
            Ptx = mul_of<T>(Ptx, sc); Pty = mul_of<T>(Pty, sc); Ptz = mul_of<T>(Ptz, sc);
        }
        dPn = sub_of<T>(Pn, r.P.x);
        dtx = sub_of<T>(Ptx, r.P.y); dty = sub_of<T>(Pty, r.P.z); dtz = sub_of<T>(Ptz, r.P.w);
    }
    const T dx = fma_of<T>(dPn, nx, dtx), dy = fma_of<T>(dPn, ny, dty), dz = fma_of<T>(dPn, nz, dtz);
    // n x dP
    const T cx = fma_of<T>(ny, dz, -mul_of<T>(nz, dy));
    const T cy = fma_of<T>(nz, dx, -mul_of<T>(nx, dz));
    const T cz = fma_of<T>(nx, dy, -mul_of<T>(ny, dx));
    va.x = fma_of<T>(-r.sa.x, dx, va.x); va.y = fma_of<T>(-r.sa.x, dy, va.y); va.z = fma_of<T>(-r.sa.x, dz, va.z);
    wa.x = fma_of<T>(-r.sa.z, cx, wa.x); wa.y = fma_of<T>(-r.sa.z, cy, wa.y); wa.z = fma_of<T>(-r.sa.z, cz, wa.z);
    if (!wall) {
        vb.x = fma_of<T>(r.sb.x, dx, vb.x); vb.y = fma_of<T>(r.sb.x, dy, vb.y); vb.z = fma_of<T>(r.sb.x, dz, vb.z);
        wb.x = fma_of<T>(-r.sb.z, cx, wb.x); wb.y = fma_of<T>(-r.sb.z, cy, wb.y); wb.z = fma_of<T>(-r.sb.z, cz, wb.z);
    }
    Pnew.x = Pn; Pnew.y = Ptx; Pnew.z = Pty; Pnew.w = Ptz;
    UpdOut o;
    const double pn = (double)Pn, px = (double)Ptx, py = (double)Pty, pz = (double)Ptz;
    o.pn = pn;
    o.pt = 0.0;
    if constexpr (sizeof(T) == 4)
        o.psq = (double)fma_of<T>(Ptz, Ptz, fma_of<T>(Pty, Pty, fma_of<T>(Ptx, Ptx, mul_of<T>(Pn, Pn))));
    else
        o.psq = __fma_rn(pz, pz, __fma_rn(py, py, __fma_rn(px, px, __dmul_rn(pn, pn))));
    o.pabs = SQ ? 0.0 : abs_of_sq<T>(o.psq);
    o.rel_ok = 0; o.bad = 0;
    if (!apply_only && crit == CD_CONV_LOCAL) {
        const double d0 = (double)dPn, d1 = (double)dtx, d2_ = (double)dty, d3 = (double)dtz;
        const double s0 = __dadd_rn(pn, (double)r.P.x), s1 = __dadd_rn(px, (double)r.P.y);
        const double s2_ = __dadd_rn(py, (double)r.P.z), s3 = __dadd_rn(pz, (double)r.P.w);
        const double d2 = __fma_rn(d3, d3, __fma_rn(d2_, d2_, __fma_rn(d1, d1, __dmul_rn(d0, d0))));
        const double s2 = __fma_rn(s3, s3, __fma_rn(s2_, s2_, __fma_rn(s1, s1, __dmul_rn(s0, s0))));
        o.rel_ok = d2 < __dmul_rn(alpha, s2);
        o.bad = !o.rel_ok && !(d2 <= __dmul_rn(__dmul_rn(alpha, ravg_prev), ravg_prev));
    }
    return o;
}

template <typename T>
__device__ __forceinline__ void wall_vel3(const CdGeom& g, const CdWork& w, int wid, typename Vec<T>::V4& vb,
                                          typename Vec<T>::V4& wb)
{
    const double* u = wall_velocity(g, w, wid);
    vb.x = (T)u[0]; vb.y = (T)u[1]; vb.z = (T)u[2]; vb.w = (T)0;
    wb.x = wb.y = wb.z = wb.w = (T)0;
}

template <typename T, bool VIEWS = false, bool DEFER = false>
__device__ __forceinline__ UpdOut apply3d(const CdGeom& g, const CdWork& w, int pos, const Rec<3, T>& r,
                                          bool apply_only, int crit, double alpha, double ravg_prev,
                                          double2 pend = make_double2(0.0, 0.0))
{
    typedef typename Vec<T>::V4 T4;
    T4* V = (T4*)w.V;
    const int ia = VIEWS ? r.vab.x : r.ab.x, ib = VIEWS ? r.vab.y : r.ab.y;
    const bool wall = !cd_is_body(g, r.ab.y);   // kinematic wall
    T4 va = V[2 * ia], wa = V[2 * ia + 1];
    T4 vb, wb;
    if (!wall) { vb = V[2 * ib]; wb = V[2 * ib + 1]; }
    else wall_vel3<T>(g, w, r.ab.y, vb, wb);
    Rec<3, T> rs = r;
    if constexpr (sizeof(T) == 8) load_static<3, T>(g, w, rs);
    const double prev = DEFER ? abs_of_pair(pend.x, pend.y) : 0.0;
    T4 Pnew;
    UpdOut o = core3d<T, DEFER>(g, rs, va, wa, vb, wb, wall, apply_only, crit, alpha, ravg_prev, Pnew);
    if constexpr (DEFER) o.pabs = prev;
    V[2 * ia] = va; V[2 * ia + 1] = wa;
    if (!wall) {
        if (r.ab.y >= g.n) {
            // a force-controlled wall moves along its normal only
            const int ax = (r.ab.y - g.n) >> 1;
            if (ax != 0) vb.x = (T)0;
            if (ax != 1) vb.y = (T)0;
            if (ax != 2) vb.z = (T)0;
            wb.x = wb.y = wb.z = (T)0;
        }
        V[2 * ib] = vb; V[2 * ib + 1] = wb;
    }
    if (!apply_only) ((T4*)w.c_P)[pos] = Pnew;
    return o;
}

template <int DIM, typename T, bool VIEWS = false, bool DEFER = false>
__device__ __forceinline__ UpdOut apply_rec(const CdGeom& g, const CdWork& w, int pos, const Rec<DIM, T>& r,
                                            bool apply_only, int crit, double alpha, double ravg_prev,
                                            double2 pend = make_double2(0.0, 0.0))
{
    if constexpr (DIM == 2)
        return apply2d<T, VIEWS, DEFER>(g, w, pos, r, apply_only, crit, alpha, ravg_prev, pend);
    else return apply3d<T, VIEWS, DEFER>(g, w, pos, r, apply_only, crit, alpha, ravg_prev, pend);
}

// Epilogue shared by both sweep kernels: impulses back to key order (FP64),
// wall forces and the solve statistics.
template <int DIM, typename T>
__device__ __forceinline__ void finish_solve(const CdGeom& g, const CdWork& w, int nc, int nb, int tid, int stride,
                                             unsigned long long& epoch, int sweeps, int converged, double resid,
                                             double ravg, double (*s_red)[3])
{
    CdCtrl* ctrl = w.ctrl;
    double wsum[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    typedef typename Vec<T>::V4 T4;
    typedef typename Vec<T>::V2 T2;
    for (int p = tid; p < nc; p += stride) {
        int c = w.perm[p];
        int2 ab = w.c_ab[p];
        double pn;
        if (DIM == 2) {
            T2 P = ((const T2*)w.c_P)[p];
            pn = (double)P.x;
            w.Pk[2 * c] = (double)P.x;
            w.Pk[2 * c + 1] = (double)P.y;
        } else {
            T4 P = ((const T4*)w.c_P)[p];
            pn = (double)P.x;
            w.Pk[4 * c] = (double)P.x;
            w.Pk[4 * c + 1] = (double)P.y;
            w.Pk[4 * c + 2] = (double)P.z;
            w.Pk[4 * c + 3] = (double)P.w;
        }
        if (ab.y >= g.n) {
            int k = ab.y - g.n;
#pragma unroll
            for (int q = 0; q < 6; ++q) if (q == k) wsum[q] += pn;
        }
    }
    {
        double a[3] = {wsum[0], wsum[1], wsum[2]};
        block_sum<3>(a, s_red);
        double b3[3] = {wsum[3], wsum[4], wsum[5]};
        block_sum<3>(b3, s_red);
        if (threadIdx.x == 0) {
            for (int q = 0; q < 3; ++q) w.wpart[q * nb + blockIdx.x] = a[q];
            for (int q = 0; q < 3; ++q) w.wpart[(3 + q) * nb + blockIdx.x] = b3[q];
        }
    }
    if (!cd_grid_sync(ctrl, nb, epoch)) return;
    if (blockIdx.x == 0) {
        // a warp a wall (one warp for all six after another, and the divisions one
        // after another, kept the last block 10 us longer)
        const int lane = threadIdx.x & 31;
        for (int q = threadIdx.x >> 5; q < 6; q += blockDim.x >> 5) {
            double x = 0.0;
            for (int b = lane; b < nb; b += 32) x += w.wpart[q * nb + b];
            x = warp_sum_nz(x);
            if (lane == 0) ctrl->wall_force[q] = x / g.dt;
        }
        if (threadIdx.x == 0) {
            ctrl->sweeps = sweeps;
            ctrl->mg_prev = sweeps + 1;
            ctrl->converged = converged;
            ctrl->residual = resid;
            ctrl->r_avg = ravg;
            ctrl->steps_done += 1;
            ctrl->total_sweeps += sweeps;
            ctrl->total_updates += (long long)sweeps * (long long)nc;
            if (sweeps > ctrl->max_sweeps_step) ctrl->max_sweeps_step = sweeps;
            if (!converged) ctrl->n_not_conv += 1;
        }
    }
}
