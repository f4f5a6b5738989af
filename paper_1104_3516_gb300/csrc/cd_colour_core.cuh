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

// The same colouring in rounds, for sets in which a thread has many contacts with
// many neighbours each, where looking again and again costs more than barriers:
// every contact counts its neighbours of higher priority, a round colours the
// contacts of its list and counts them off at their neighbours of lower priority,
// and those left with none make the next list.  Scratch: the colour repair's
// arrays (rep_flag the counts, rep_list and rep_path the lists of even and odd
// rounds) and round_cnt[r % 3], the length of round r's list (cleared two rounds
// ahead).
__device__ __forceinline__ bool jp_higher(const CdWork& w, const unsigned long long* prio, int d, int c,
                                          unsigned long long pc, unsigned long long kc)
{
    const unsigned long long pd = prio[d];
    if (pd != pc) return pd > pc;
    const int2 dd = w.pairs[d];
    return cd_key(dd.x, dd.y) < kc;
}

// Appends each lane's up to N entries c[u] (take[u]) with one atomic a warp.
template <int N>
__device__ __forceinline__ void jp_append(int* list, int* len, const int (&c)[N], const bool (&take)[N])
{
    const int lane = threadIdx.x & 31;
    int k = 0;
#pragma unroll
    for (int u = 0; u < N; ++u) k += take[u] ? 1 : 0;
    int incl = k;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    if (total == 0) return;
    int base = 0;
    if (lane == 31) base = atomicAdd(len, total);
    base = __shfl_sync(0xffffffffu, base, 31) + incl - k;
#pragma unroll
    for (int u = 0; u < N; ++u)
        if (take[u]) list[base++] = c[u];
}

// (priorities set, colours -1, round_cnt 0, behind a barrier)
template <typename SYNC>
__device__ __forceinline__ bool jp_rounds(const CdGeom& g, const CdWork& w, int nc, const unsigned long long* prio,
                                          SYNC& sync)
{
    CdCtrl* ctrl = w.ctrl;
    const int stride = gridDim.x * blockDim.x, lane = threadIdx.x & 31;
    const int warp0 = blockIdx.x * blockDim.x + (int)(threadIdx.x & ~31u);
    int* const cnt = w.rep_flag;
    for (int c0 = warp0; c0 < nc; c0 += stride) {
        const int c[1] = {c0 + lane};
        int k = 0;
        if (c[0] < nc) {
            const unsigned long long pc = prio[c[0]];
            const int2 ab = w.pairs[c[0]];
            const unsigned long long kc = cd_key(ab.x, ab.y);
            for (int side = 0; side < 2; ++side) {
                const int q = side ? ab.y : ab.x;
                if (!cd_is_body(g, q)) continue;
                const int f0 = w.p2c_off[q], f1 = w.p2c_off[q + 1];
                for (int t = f0; t < f1; t += 4) {
                    int d[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) d[u] = (t + u < f1) ? w.p2c[t + u] : c[0];
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (d[u] != c[0] && jp_higher(w, prio, d[u], c[0], pc, kc)) ++k;
                }
            }
            cnt[c[0]] = k;
        }
        const bool free[1] = {c[0] < nc && k == 0};
        jp_append<1>(w.rep_list, &w.round_cnt[0], c, free);
    }
    if (!sync()) return false;
    int top = 0;
    for (int round = 0;; ++round) {   // (ends with the longest chain of priorities, at most nc)
        // (selected, not indexed: an indexed pair of pointers lives in local memory)
        int* const list = (round & 1) ? w.rep_path : w.rep_list;
        int* const next = (round & 1) ? w.rep_list : w.rep_path;
        const int len = cd_ld_volatile_int(&w.round_cnt[round % 3]);
        if (len == 0) break;
        if (warp0 == 0 && lane == 0) w.round_cnt[(round + 2) % 3] = 0;
        for (int i0 = warp0; i0 < len; i0 += stride) {
            const int c = (i0 + lane < len) ? list[i0 + lane] : -1;
            int2 ab = make_int2(0, 0);
            unsigned long long pc = 0ULL, kc = 0ULL, used = 0ULL;
            if (c >= 0) {
                pc = prio[c];
                ab = w.pairs[c];
                kc = cd_key(ab.x, ab.y);
            }
            // the colours of the neighbours of higher priority (all final), and one off for
            // those of lower (which read c's colour behind the next barrier)
            for (int side = 0; side < 2; ++side) {
                const int q = side ? ab.y : ab.x;
                const bool on = c >= 0 && cd_is_body(g, q);
                const int f0 = on ? w.p2c_off[q] : 0, f1 = on ? w.p2c_off[q + 1] : 0;
                const int most = __reduce_max_sync(0xffffffffu, f1 - f0);
                for (int t = 0; t < most; t += 4) {
                    int d[4], v[4];
                    bool hi[4], lo[4], rel[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) d[u] = (f0 + t + u < f1) ? w.p2c[f0 + t + u] : c;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        hi[u] = d[u] != c && jp_higher(w, prio, d[u], c, pc, kc);
                        lo[u] = d[u] != c && !hi[u];
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        v[u] = hi[u] ? cd_ld_volatile_int(&w.colour[d[u]]) : (lo[u] ? atomicSub(&cnt[d[u]], 1) : 0);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (hi[u] && v[u] >= 0) used |= 1ULL << v[u];
                        rel[u] = lo[u] && v[u] == 1;
                    }
                    jp_append<4>(next, &w.round_cnt[(round + 1) % 3], d, rel);
                }
            }
            if (c >= 0) {
                const int k = (used == ~0ULL) ? 64 : __ffsll((long long)~used) - 1;
                if (k >= CD_KMAX) atomicCAS(&ctrl->error, CDE_NONE, CDE_COLOURS);
                else {
                    *(volatile int*)&w.colour[c] = k;
                    top = max(top, k + 1);
                }
            }
        }
        if (!sync()) return false;
    }
    top = __reduce_max_sync(0xffffffffu, top);
    if (lane == 0 && top > 0) atomicMax(&ctrl->ncolours, top);
    return sync();
}

// Where rounds are faster: more than nine contacts a thread, with three a body or
// more (of a gas most contacts have hardly a neighbour to wait for).  Colouring
// and order, tries / rounds: 200,000 packed discs (447,000 contacts, 152 x 512
// threads) 0.41 / 0.48 ms, 400,000 0.69 / 0.56, 1,000,000 1.44 / 0.98; a lattice of
// spheres with 11 contacts each, 549,000 contacts 1.89 / 2.29, 1,108,000 3.48 /
// 2.61, 5,595,000 19.7 / 7.4; 512 squeezed packings of 38 colours 61 / 21; a gas of a
// million spheres 0.39 / 0.46, of four 1.48 / 1.84.
__device__ __forceinline__ bool jp_in_rounds(const CdGeom& g, int nc, int threads)
{
    return nc > 9 * threads && nc > g.n + (g.n >> 1);
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
    if (tid == 0) ctrl->ncolours = w.round_cnt[0] = w.round_cnt[1] = w.round_cnt[2] = 0;
    if (!sync()) return false;
    if (jp_in_rounds(g, nc, stride)) return jp_rounds(g, w, nc, prio, sync);
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
