// cd_flow_core.cuh -- what the dataflow kernels share: tagged records, tagged
// block sums, bounded waits.
#pragma once

#include "cd_sweep_core.cuh"

// ---------------------------------------------------------------------------
// Tagged velocity records.  A record is made of 64-bit elements, each 48 bits
// of velocity and a 16-bit tag, the number of updates its body has had (modulo
// 2^16).  Every element says by itself which update it belongs to, so a reader
// that finds the tag it expects in all of them has that update's velocities:
// no fence, no flag beside the data.  (A reader is at most one pass behind a
// writer: 64 updates, 65 of a particle that domains share.)  Three numbers make a group: FP64 four elements
// (one 256-bit access), FP32 two (one 128-bit access); 2D has one group
// (v_x, v_y, omega), 3D two (v, omega).
// ---------------------------------------------------------------------------
typedef unsigned long long u64;
template <typename T> struct FlowGroup;
template <> struct FlowGroup<double> { static constexpr int N = 4; };
template <> struct FlowGroup<float> { static constexpr int N = 2; };

__device__ __forceinline__ void flow_load(const u64* p, u64 (&e)[4])
{
    asm volatile("ld.relaxed.gpu.global.v4.b64 {%0, %1, %2, %3}, [%4];"
                 : "=l"(e[0]), "=l"(e[1]), "=l"(e[2]), "=l"(e[3]) : "l"(p) : "memory");
}
__device__ __forceinline__ void flow_load(const u64* p, u64 (&e)[2])
{
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(e[0]), "=l"(e[1]) : "l"(p) : "memory");
}
__device__ __forceinline__ void flow_store(u64* p, const u64 (&e)[4])
{
    asm volatile("st.relaxed.gpu.global.v4.b64 [%0], {%1, %2, %3, %4};"
                 :: "l"(p), "l"(e[0]), "l"(e[1]), "l"(e[2]), "l"(e[3]) : "memory");
}
__device__ __forceinline__ void flow_store(u64* p, const u64 (&e)[2])
{
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" :: "l"(p), "l"(e[0]), "l"(e[1]) : "memory");
}

__device__ __forceinline__ u64 flow_pair(unsigned lo, unsigned hi) { return ((u64)hi << 32) | (u64)lo; }
__device__ __forceinline__ unsigned flow_lo(u64 x) { return (unsigned)x; }
__device__ __forceinline__ unsigned flow_hi(u64 x) { return (unsigned)(x >> 32); }
__device__ __forceinline__ unsigned flow_tag(u64 e) { return (unsigned)(e >> 48); }

// Three FP64 numbers: their low 48 bits in elements 0 to 2, their top 16 bits
// together in element 3.
__device__ __forceinline__ void flow_pack(double a, double b, double c, unsigned tag, u64 (&e)[4])
{
    const u64 x = (u64)__double_as_longlong(a), y = (u64)__double_as_longlong(b), z = (u64)__double_as_longlong(c);
    e[0] = flow_pair(flow_lo(x), __byte_perm(flow_hi(x), tag, 0x5410));
    e[1] = flow_pair(flow_lo(y), __byte_perm(flow_hi(y), tag, 0x5410));
    e[2] = flow_pair(flow_lo(z), __byte_perm(flow_hi(z), tag, 0x5410));
    e[3] = flow_pair(__byte_perm(flow_hi(x), flow_hi(y), 0x7632), __byte_perm(flow_hi(z), tag, 0x5432));
}
__device__ __forceinline__ void flow_unpack(const u64 (&e)[4], double& a, double& b, double& c)
{
    a = __hiloint2double((int)__byte_perm(flow_hi(e[0]), flow_lo(e[3]), 0x5410), (int)flow_lo(e[0]));
    b = __hiloint2double((int)__byte_perm(flow_hi(e[1]), flow_lo(e[3]), 0x7610), (int)flow_lo(e[1]));
    c = __hiloint2double((int)__byte_perm(flow_hi(e[2]), flow_hi(e[3]), 0x5410), (int)flow_lo(e[2]));
}
// Three FP32 numbers: a and b whole, c in two halves.
__device__ __forceinline__ void flow_pack(float a, float b, float c, unsigned tag, u64 (&e)[2])
{
    const unsigned z = __float_as_uint(c);
    e[0] = flow_pair(__float_as_uint(a), __byte_perm(z, tag, 0x5410));
    e[1] = flow_pair(__float_as_uint(b), __byte_perm(z, tag, 0x5432));
}
__device__ __forceinline__ void flow_unpack(const u64 (&e)[2], float& a, float& b, float& c)
{
    a = __uint_as_float(flow_lo(e[0]));
    b = __uint_as_float(flow_lo(e[1]));
    c = __uint_as_float(__byte_perm(flow_hi(e[0]), flow_hi(e[1]), 0x5410));
}

// A body's record.
template <int DIM, typename T>
struct FlowBody {
    static constexpr int G = (DIM == 2) ? 1 : 2;
    static constexpr int N = FlowGroup<T>::N;
    u64 e[G][N];
    __device__ __forceinline__ void load(const u64* p)
    {
#pragma unroll
        for (int q = 0; q < G; ++q) flow_load(p + q * N, e[q]);
    }
    __device__ __forceinline__ void store(u64* p) const
    {
#pragma unroll
        for (int q = 0; q < G; ++q) flow_store(p + q * N, e[q]);
    }
    __device__ __forceinline__ bool has(unsigned tag) const
    {
        unsigned off = 0u;
#pragma unroll
        for (int q = 0; q < G; ++q)
#pragma unroll
            for (int j = 0; j < N; ++j) off |= flow_hi(e[q][j]) ^ (tag << 16);
        return (off >> 16) == 0u;
    }
    __device__ __forceinline__ void pack(const typename Vec<T>::V4& v, const typename Vec<T>::V4& o, unsigned tag)
    {
        flow_pack(v.x, v.y, v.z, tag, e[0]);
        if constexpr (DIM == 3) flow_pack(o.x, o.y, o.z, tag, e[1]);
    }
    __device__ __forceinline__ void unpack(typename Vec<T>::V4& v, typename Vec<T>::V4& o) const
    {
        flow_unpack(e[0], v.x, v.y, v.z);
        v.w = (T)0;
        if constexpr (DIM == 3) {
            flow_unpack(e[1], o.x, o.y, o.z);
            o.w = (T)0;
        }
    }
};

// A block's sum of residual terms, tagged with its pass.
struct FlowSum { u64 e[2]; };
__device__ __forceinline__ void flow_sum_store(FlowSum* p, double x, unsigned tag)
{
    // 48 bits and 16 bits of the sum, each with a tag
    const u64 b = (u64)__double_as_longlong(x);
    const u64 e[2] = {(b & 0xffffffffffffULL) | ((u64)tag << 48), (b >> 48) | ((u64)tag << 48)};
    flow_store(p->e, e);
}
__device__ __forceinline__ bool flow_sum_is(const u64 (&e)[2], unsigned tag)
{
    return flow_tag(e[0]) == (tag & 0xffffu) && flow_tag(e[1]) == (tag & 0xffffu);
}
__device__ __forceinline__ double flow_sum_of(const u64 (&e)[2])
{
    return __longlong_as_double((long long)((e[0] & 0xffffffffffffULL) | (e[1] << 48)));
}

__device__ __forceinline__ int flow_ld(const int* p) { return *(volatile const int*)p; }

// A bounded wait: gives up CD_WAIT_NS after its first look at the clock, or
// when another block has flagged an error.
struct FlowBound {
    unsigned spins = 0;
    u64 t0 = 0;
    __device__ __forceinline__ bool look(CdCtrl* ctrl)
    {
        if (t0 == 0) t0 = cd_globaltimer();
        else if (cd_globaltimer() - t0 > CD_WAIT_NS) {
            atomicCAS(&ctrl->error, CDE_NONE, CDE_TIMEOUT);
            return false;
        }
        return cd_ld_volatile_int(&ctrl->error) == CDE_NONE;
    }
    __device__ __forceinline__ bool go(CdCtrl* ctrl) { return (++spins & 255u) != 0u || look(ctrl); }
};

// Looks again at the records at pa and pb (null: none) until they carry their
// tags (the caller has looked once: ra, rb); the lanes of a warp leave
// together.  False when a wait gave up (this one, or another of the block: *gave_up).
template <int DIM, typename T>
__device__ __forceinline__ bool flow_wait(CdCtrl* ctrl, int* gave_up, const u64* pa, unsigned ta, const u64* pb,
                                          unsigned tb, FlowBody<DIM, T>& A, FlowBody<DIM, T>& B, bool ra, bool rb)
{
    FlowBound bound;
    while (!__all_sync(0xffffffffu, ra && rb)) {
        if (!ra) A.load(pa);
        if (!rb) B.load(pb);
        ra = ra || A.has(ta);
        rb = rb || B.has(tb);
        if ((++bound.spins & 63u) == 0u && !__all_sync(0xffffffffu, bound.look(ctrl) && !flow_ld(gave_up))) {
            *(volatile int*)gave_up = 1;
            return false;
        }
    }
    return true;
}

// The sum of N values >= 0 a lane over the warp (in every lane), as integers of
// 128 bits that share the largest exponent, added a lane and then by limbs of 25
// bits: of each term what is below 2^-116 of the largest one's binade is cut
// off, and the sum is rounded once.  (Near the ends of the range FP64 adds.)  The
// FP64 pipe takes 64
// cycles an instruction, more while the workers use it; a pass's sums and test
// took 9,000 cycles on it, longer than a pass of two colours (10,000 discs in
// pyramids, 150 sweeps: 875 us, now 640).
template <int N>
__device__ __forceinline__ double flow_sum_warp(const double (&v)[N])
{
    typedef unsigned __int128 u128;
    unsigned top = 0;
#pragma unroll
    for (int u = 0; u < N; ++u) top = max(top, (unsigned)((u64)__double_as_longlong(v[u]) >> 32));
    top = __reduce_max_sync(0xffffffffu, top);
    if (top == 0u) top = __any_sync(0xffffffffu, [&]() { u64 o = 0; for (int u = 0; u < N; ++u) o |= (u64)__double_as_longlong(v[u]); return o != 0; }());
    if (top == 0u) return 0.0;
    const int em = (int)(top >> 20);
    if (em < 128 || em > 2032) {   // near the ends of the range, infinite, NaN
        double x = 0.0;
        for (int u = 0; u < N; ++u) x += v[u];
        return warp_sum(x);
    }
    u128 t = 0;   // bit 116: 2^(em - 1023)
#pragma unroll
    for (int u = 0; u < N; ++u) {
        const u64 b = (u64)__double_as_longlong(v[u]);
        const int e = (int)(b >> 52), d = em - e;
        const u64 m = (b & 0xfffffffffffffULL) | (1ULL << 52);
        if (e > 0 && d < 117) t += ((u128)m << 64) >> d;
    }
    u128 s = 0;
#pragma unroll
    for (int q = 4; q >= 0; --q)
        s = (s << 25) + __reduce_add_sync(0xffffffffu, (unsigned)(t >> (25 * q)) & 0x1ffffffu);
    const u64 hi = (u64)(s >> 64);   // (not 0: the largest term's bit 52)
    const int z = __clzll((long long)hi);
    s <<= z;
    const u64 m = (u64)(s >> 75) + ((u64)(s >> 74) & 1ULL);
    return __longlong_as_double((long long)(((u64)(em + 11 - z - 1) << 52) + m));
}
