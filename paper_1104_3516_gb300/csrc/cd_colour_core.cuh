// cd_colour_core.cuh -- the pieces of the colouring and of the colour ordering
// that the colouring kernels share.
#pragma once

#include <type_traits>

#include "cd_internal.cuh"

// Jones-Plassmann colouring without rounds.  A contact's colour depends on its
// neighbours of higher priority alone (contacts sharing a body), and a colour
// once written is final: a thread goes over its contacts again and again, and
// gives each one the smallest colour that no higher-priority neighbour has as
// soon as all of those are coloured.  A colour is its own flag, so reading it
// needs neither fence nor barrier, and a step along the longest chain of
// priorities takes one look (about 1,500 cycles) instead of a round of
// dependent loads and atomics behind a barrier (11,000).  No thread waits for
// a single contact, so the contact of the highest priority left can always be
// coloured.  The result is the greedy colouring whatever the timing.

// The colour of contact c, or -1 while a higher-priority neighbour has none.
// Eight neighbours at a time, their loads in flight together.
__device__ __forceinline__ int jp_try(const CdGeom& g, const CdWork& w, const unsigned long long* __restrict__ prio,
                                      int c)
{
    const int2 ab = w.pairs[c];
    const unsigned long long pc = prio[c];
    const int fa = w.p2c_off[ab.x], la = w.p2c_off[ab.x + 1] - fa;
    int fb = 0, lb = 0;
    if (cd_is_body(g, ab.y)) { fb = w.p2c_off[ab.y]; lb = w.p2c_off[ab.y + 1] - fb; }
    unsigned long long used = 0ULL;
    for (int t = 0; t < la + lb; t += 8) {
        int d[8], v[8];
        unsigned long long pd[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            d[u] = (t + u < la + lb) ? w.p2c[(t + u < la) ? fa + t + u : fb + t + u - la] : c;
#pragma unroll
        for (int u = 0; u < 8; ++u) pd[u] = prio[d[u]];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            bool higher = pd[u] > pc;
            if (pd[u] == pc && d[u] != c) {   // ties by ascending key
                const int2 dd = w.pairs[d[u]];
                higher = cd_key(dd.x, dd.y) < cd_key(ab.x, ab.y);
            }
            v[u] = higher ? cd_ld_volatile_int(&w.colour[d[u]]) : 64;
        }
        bool wait = false;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            wait = wait || v[u] < 0;
            if (v[u] >= 0 && v[u] < 64) used |= 1ULL << v[u];
        }
        if (wait) return -1;
    }
    return (used == ~0ULL) ? 64 : __ffsll((long long)~used) - 1;
}

// All contacts; `sync` is the barrier of the blocks (false: it gave up).
template <typename SYNC>
__device__ __forceinline__ bool jp_colour(const CdGeom& g, const CdWork& w, int nc, unsigned long long* prio,
                                          SYNC& sync)
{
    CdCtrl* ctrl = w.ctrl;
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int stride = gridDim.x * blockDim.x;
    for (int c = tid; c < nc; c += stride) {
        int2 ab = w.pairs[c];
        unsigned long long h;
        if (g.npk > 1) {
            // a packing of a batch is coloured with its own seed and local
            // ids (walls n_b + k), exactly as if it were a system alone
            const CdPack& P = w.pk[w.pack_of[ab.x]];
            const int al = ab.x - P.first;
            const int bl = (ab.y < g.n) ? ab.y - P.first : P.count + (ab.y - g.n) % 6;
            h = cd_splitmix64(P.seed ^ cd_key(al, bl));
        } else {
            h = cd_splitmix64(g.seed ^ cd_key(ab.x, ab.y));
        }
        // largest degree first (contacts of both ends, capped at 255), then the hash
        unsigned long long ds = (unsigned long long)(w.p2c_off[ab.x + 1] - w.p2c_off[ab.x]);
        if (cd_is_body(g, ab.y)) ds += (unsigned long long)(w.p2c_off[ab.y + 1] - w.p2c_off[ab.y]);
        if (ds > 255ULL) ds = 255ULL;
        prio[c] = (ds << 56) | (h >> 8);
        w.colour[c] = -1;
    }
    if (tid == 0) ctrl->ncolours = 0;
    if (!sync()) return false;
    int top = 0;
    unsigned long long t0 = 0ULL;
    bool on = true;
    int first = tid;   // the thread's contacts before this one are coloured
    for (unsigned pass = 1; first < nc && on; ++pass) {
        int left = nc;
        for (int c = first; c < nc; c += stride) {
            if (w.colour[c] >= 0) continue;   // written by this thread
            const int k = jp_try(g, w, prio, c);
            if (k < 0) {
                left = min(left, c);
            } else if (k >= CD_KMAX) {
                atomicCAS(&ctrl->error, CDE_NONE, CDE_COLOURS);
                left = min(left, c);
            } else {
                *(volatile int*)&w.colour[c] = k;
                top = max(top, k + 1);
            }
        }
        first = left;
        if ((pass & 15u) == 0u) {
            // bounded, and ended by an error elsewhere
            if (t0 == 0ULL) t0 = cd_globaltimer();
            else if (cd_globaltimer() - t0 > CD_WAIT_NS) atomicCAS(&ctrl->error, CDE_NONE, CDE_TIMEOUT);
            on = cd_ld_volatile_int(&ctrl->error) == CDE_NONE;
        }
    }
    __syncwarp();
    top = __reduce_max_sync(0xffffffffu, top);   // one atomic per warp
    if ((threadIdx.x & 31) == 0 && top > 0) atomicMax(&ctrl->ncolours, top);
    return sync();
}

// The repair runs one warp per packing: every step is sequential, but the
// lanes read a body's contact list together, so a step costs a few L2 round
// trips instead of one per contact of the body.  All lanes follow the same
// control flow; lane 0 writes.

// Colours below t that body x has on no contact other than c (all of them
// for a wall that is not a body).
__device__ __forceinline__ unsigned long long rep_free(const CdGeom& g, const CdWork& w, int x, int c, int t)
{
    const unsigned long long all = (1ULL << t) - 1ULL;
    if (!cd_is_body(g, x)) return all;
    const int lane = threadIdx.x & 31;
    const int f0 = w.p2c_off[x], f1 = w.p2c_off[x + 1];
    unsigned long long used = 0ULL;
    for (int f = f0; f < f1; f += 32) {
        unsigned long long bit = 0ULL;
        if (f + lane < f1) {
            const int d = w.p2c[f + lane];
            const int k = w.colour[d];
            if (d != c && k >= 0 && k < t) bit = 1ULL << k;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) bit |= __shfl_xor_sync(0xffffffffu, bit, o);
        used |= bit;
    }
    return all & ~used;
}

// Body x's contact of colour cur (at most one in a proper colouring), or -1.
__device__ __forceinline__ int rep_find(const CdWork& w, int x, int cur)
{
    const int lane = threadIdx.x & 31;
    const int f0 = w.p2c_off[x], f1 = w.p2c_off[x + 1];
    for (int f = f0; f < f1; f += 32) {
        int d = -1;
        if (f + lane < f1) {
            const int dd = w.p2c[f + lane];
            if (w.colour[dd] == cur) d = dd;
        }
        const unsigned hit = __ballot_sync(0xffffffffu, d >= 0);
        if (hit) return __shfl_sync(0xffffffffu, d, __ffs(hit) - 1);
    }
    return -1;
}

// Whether the repair of the highest colour is tried: ncb contacts, highest
// colour t (held by `top` of them), at most dmax contacts at a body.
__device__ __forceinline__ bool rep_wanted(int ncb, int t, int dmax, int top)
{
    if (ncb <= 0 || t <= 0 || t > 63 || t + 1 <= dmax) return false;
    int limit = ncb / 256;
    if (limit > 1024) limit = 1024;
    if (limit < 1) limit = 1;
    return top <= limit;
}

// The contacts rep_list[l0 .. l1) of colour t, one warp; ncb contacts in the
// packing, `path` room for as many.
__device__ __forceinline__ void rep_run(const CdGeom& g, const CdWork& w, int t, int l0, int l1, int ncb, int* path)
{
    const int lane = threadIdx.x & 31;
    for (int l = l0; l < l1; ++l) {
        const int c = w.rep_list[l];
        const int2 uv = w.pairs[c];
        const int u = uv.x, v = uv.y;
        const unsigned long long mu = rep_free(g, w, u, c, t), mv = rep_free(g, w, v, c, t);
        if (mu & mv) {
            if (lane == 0) w.colour[c] = __ffsll((long long)(mu & mv)) - 1;
            __syncwarp();
            continue;
        }
        if (!cd_is_body(g, v)) continue;
        bool done = false;
        for (int a = 0; a < t && !done; ++a) {
            if (!((mu >> a) & 1ULL)) continue;
            for (int bb = 0; bb < t && !done; ++bb) {
                if (!((mv >> bb) & 1ULL)) continue;
                int len = 0, x = v, cur = a;
                bool fail = false;
                for (;;) {
                    const int e = rep_find(w, x, cur);
                    if (e < 0) break;
                    const int2 pe = w.pairs[e];
                    const int y = (pe.x == x) ? pe.y : pe.x;
                    if (lane == 0) path[len] = e;
                    ++len;
                    if (y == u) { fail = true; break; }
                    if (!cd_is_body(g, y)) break;
                    x = y;
                    cur = (cur == a) ? bb : a;
                    if (len >= ncb) { fail = true; break; }
                }
                __syncwarp();
                if (fail) continue;
                for (int i = lane; i < len; i += 32) {
                    const int e = path[i];
                    w.colour[e] = (w.colour[e] == a) ? bb : a;
                }
                if (lane == 0) w.colour[c] = a;
                __syncwarp();
                done = true;
            }
        }
    }
}

// Contact c's record at colour-order position pos, in the sweep's real type.
template <int DIM, typename T>
__device__ __forceinline__ void colour_record(const CdGeom& g, const CdWork& w, int c, int pos)
{
    w.perm[pos] = c;
    int2 ab = w.pairs[c];
    w.c_ab[pos] = ab;
    double b = __ddiv_rn(w.gap[c], g.dt);
    if (DIM == 2) {
        typedef typename std::conditional<sizeof(T) == 8, double4_32a, float4>::type T4;
        typedef typename std::conditional<sizeof(T) == 8, double2, float2>::type T2;
        T4 geo;
        geo.x = (T)w.nrm[3 * c];
        geo.y = (T)w.nrm[3 * c + 1];
        geo.z = (T)b;
        geo.w = (T)w.mn[c];
        ((T4*)w.c_geo)[pos] = geo;
        ((T*)w.c_m)[pos] = (T)w.mt[c];
        T2 P;
        P.x = (T)w.Pk[2 * c];
        P.y = (T)w.Pk[2 * c + 1];
        ((T2*)w.c_P)[pos] = P;
    } else {
        typedef typename std::conditional<sizeof(T) == 8, double4_32a, float4>::type T4;
        typedef typename std::conditional<sizeof(T) == 8, double2, float2>::type T2;
        T4 geo;
        geo.x = (T)w.nrm[3 * c];
        geo.y = (T)w.nrm[3 * c + 1];
        geo.z = (T)w.nrm[3 * c + 2];
        geo.w = (T)b;
        ((T4*)w.c_geo)[pos] = geo;
        T2 m;
        m.x = (T)w.mn[c];
        m.y = (T)w.mt[c];
        ((T2*)w.c_m)[pos] = m;
        T4 P;
        P.x = (T)w.Pk[4 * c];
        P.y = (T)w.Pk[4 * c + 1];
        P.z = (T)w.Pk[4 * c + 2];
        P.w = (T)w.Pk[4 * c + 3];
        ((T4*)w.c_P)[pos] = P;
    }
}
