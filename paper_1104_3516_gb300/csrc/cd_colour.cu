// cd_colour.cu -- colouring of the contact graph and the colour ordering.
//
// The paper updates contacts one by one in random order (Sec. 2.1).  On the
// GPU the same nonlinear Gauss-Seidel runs in a colour order: contacts that
// share no particle are independent, so one colour class is updated in
// parallel and every freshly computed impulse is seen by the later colours.
//
// Colouring: Jones-Plassmann with priority (d_a + d_b) * 2^56 +
// (splitmix64(seed ^ key) >> 8), d the contacts of a particle (largest degree
// first, which needs one colour fewer than a random order on dense piles),
// ties by ascending key.  A contact takes the smallest colour not used by any
// higher-priority neighbour once all of those are coloured; the fixed point
// equals the greedy colouring in descending priority, so the result does not
// depend on scheduling.  Walls never conflict.
//
// Ordering: stable partition of the key-ordered contacts by colour (chunk
// histograms, one exclusive scan, a rank within the chunk from warp match
// masks), then the contact data is gathered into colour order in the sweep's
// real type.
#include "cd_colour_core.cuh"

__global__ void k_p2c_count(CdGeom g, CdWork w)
{
    CdCtrl* ctrl = w.ctrl;
    if (ctrl->skip) return;
    int nc = ctrl->nc;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x) {
        int2 ab = w.pairs[c];
        atomicAdd(&w.p2c_cnt[ab.x], 1);
        if (cd_is_body(g, ab.y)) atomicAdd(&w.p2c_cnt[ab.y], 1);
    }
}

__global__ void k_p2c_fill(CdGeom g, CdWork w)
{
    CdCtrl* ctrl = w.ctrl;
    if (ctrl->skip) return;
    int nc = ctrl->nc;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x) {
        int2 ab = w.pairs[c];
        int s = atomicAdd(&w.p2c_fill[ab.x], 1);
        w.p2c[w.p2c_off[ab.x] + s] = c;
        if (cd_is_body(g, ab.y)) {
            s = atomicAdd(&w.p2c_fill[ab.y], 1);
            w.p2c[w.p2c_off[ab.y] + s] = c;
        }
    }
}

// Each particle's contact list in ascending key order (the atomic fill leaves
// it in arrival order); makes every later per-particle accumulation
// deterministic.
__global__ void k_p2c_sort(CdGeom g, CdWork w)
{
    if (w.ctrl->skip) return;
    const int nbody = g.n + (g.dyn_walls ? 6 : 0);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nbody; i += gridDim.x * blockDim.x) {
        int b = w.p2c_off[i], e = w.p2c_off[i + 1];
        for (int k = b + 1; k < e; ++k) {
            int v = w.p2c[k];
            int j = k - 1;
            while (j >= b && w.p2c[j] > v) { w.p2c[j + 1] = w.p2c[j]; --j; }
            w.p2c[j + 1] = v;
        }
    }
}

// Persistent cooperative kernel.
__global__ void __launch_bounds__(CD_SWEEP_THREADS) k_jp(CdGeom g, CdWork w, unsigned long long* prio)
{
    CdCtrl* ctrl = w.ctrl;
    if (ctrl->skip) return;
    unsigned long long epoch = 0;
    const unsigned long long nb = gridDim.x;
    auto sync = [&]() { return cd_grid_sync(ctrl, nb, epoch); };
    jp_colour(g, w, ctrl->nc, prio, sync);
}

// ---------------------------------------------------------------------------
// Repair of the highest colour (Kempe chains; the recolouring step of the
// classical proof of Vizing's theorem, used as a heuristic).  For each
// packing (a plain system is one): if its greedy colouring has a colour more
// than its busiest body has contacts, and that top colour T holds at most
// max(1, min(1024, nc_b / 256)) contacts, one warp visits them in key
// order.  Contact c = (u, v) takes the smallest colour below T that neither
// u nor v has; failing that, for a free at u and b free at v (ascending),
// the path leaving v on its colour-a contact and alternating a, b is
// followed to its end (a body without the next colour, or a wall); unless it
// reaches u, a and b are swapped along it and c takes a.  Fewer colours mean
// fewer grid barriers per sweep.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int rep_pack_of(const CdGeom& g, const CdWork& w, int body)
{
    return (g.npk > 1) ? w.pack_of[body] : 0;
}

__global__ void k_rep_init(CdGeom g, CdWork w)
{
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < g.npk; b += gridDim.x * blockDim.x) {
        w.rep_top[b] = -1;
        w.rep_dmax[b] = 0;
    }
}

// atomicMax of v into dst[key], one atomic per run of lanes with the same key
// (the plain system's single packing would otherwise serialise every
// contact on one address).
__device__ __forceinline__ void warp_atomic_max(int* dst, int key, int v, bool active)
{
    const unsigned grp = __match_any_sync(0xffffffffu, active ? key : -1);
    const int m = __reduce_max_sync(grp, active ? v : -1);
    if (active && (threadIdx.x & 31) == __ffs(grp) - 1) atomicMax(&dst[key], m);
}

// The largest v >= -1 of the block, one atomicMax for it.
__device__ __forceinline__ void block_atomic_max(int* dst, int v)
{
    __shared__ int s_max;
    if (threadIdx.x == 0) s_max = -1;
    __syncthreads();
    v = __reduce_max_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_max, v);
    __syncthreads();
    if (threadIdx.x == 0) atomicMax(dst, s_max);
}

// The highest colour and the most contacts at a body, of each packing.  (A
// plain system knows the colour already, and takes an atomic a block: one a
// warp on one address took 25 us of a million spheres' step.)
__global__ void k_rep_scan_colours(CdGeom g, CdWork w)
{
    if (w.ctrl->skip) return;
    const int nc = w.ctrl->nc;
    const int nbody = g.n + (g.dyn_walls ? 6 : 0);
    const int st = gridDim.x * blockDim.x;
    if (g.npk == 1) {
        int d = 0;
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nbody; i += st)
            d = max(d, w.p2c_off[i + 1] - w.p2c_off[i]);
        block_atomic_max(w.rep_dmax, d);
        if (blockIdx.x == 0 && threadIdx.x == 0) w.rep_top[0] = w.ctrl->ncolours - 1;
        return;
    }
    // whole warps iterate together (the warp collectives need every lane)
    for (int c0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31); c0 < nc; c0 += st) {
        const int c = c0 + (threadIdx.x & 31);
        const bool on = c < nc;
        warp_atomic_max(w.rep_top, on ? rep_pack_of(g, w, w.pairs[c].x) : 0, on ? w.colour[c] : -1, on);
    }
    for (int i0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < nbody; i0 += st) {
        const int i = i0 + (threadIdx.x & 31);
        const bool on = i < nbody;
        const int pk = (on && i < g.n) ? rep_pack_of(g, w, i) : 0;
        warp_atomic_max(w.rep_dmax, pk, on ? w.p2c_off[i + 1] - w.p2c_off[i] : 0, on);
    }
}

// Flags over the whole capacity (the scan runs over cap + 1 entries).
__global__ void k_rep_flag(CdGeom g, CdWork w)
{
    if (w.ctrl->skip) return;
    const int nc = w.ctrl->nc;
    // up to nc: the scan of the flags reads the live contacts only
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c <= nc; c += gridDim.x * blockDim.x) {
        int f = 0;
        if (c < nc) {
            const int t = w.rep_top[rep_pack_of(g, w, w.pairs[c].x)];
            f = (t > 0 && w.colour[c] == t) ? 1 : 0;
        }
        w.rep_flag[c] = f;
    }
}

__global__ void k_rep_fill(CdWork w)
{
    if (w.ctrl->skip) return;
    const int nc = w.ctrl->nc;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x)
        if (w.rep_flag[c]) w.rep_list[w.rep_pos[c]] = c;
}

// One warp per packing.
__global__ void k_rep_run(CdGeom g, CdWork w)
{
    if (w.ctrl->skip || w.ctrl->error != CDE_NONE) return;   // e.g. an uncoloured contact
    const int nc = w.ctrl->nc;
    const int b = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (b >= g.npk) return;
    const int c0 = (g.npk > 1) ? w.pk_coff[b] : 0, c1 = (g.npk > 1) ? w.pk_coff[b + 1] : nc;
    const int t = w.rep_top[b], l0 = w.rep_pos[c0], l1 = w.rep_pos[c1];
    if (rep_wanted(c1 - c0, t, w.rep_dmax[b], l1 - l0)) rep_run(g, w, t, l0, l1, c1 - c0, w.rep_path + c0);
}

// Whether the repair ran on the plain system (whose colours then are counted anew).
__device__ __forceinline__ bool rep_ran(const CdWork& w, int nc)
{
    return rep_wanted(nc, w.rep_top[0], w.rep_dmax[0], w.rep_pos[nc] - w.rep_pos[0]);
}

__global__ void k_rep_ncolours_reset(CdGeom g, CdWork w)
{
    if (w.ctrl->skip) return;
    if (g.npk > 1 || rep_ran(w, w.ctrl->nc)) w.ctrl->ncolours = 0;
}

__global__ void k_rep_ncolours(CdGeom g, CdWork w)
{
    if (w.ctrl->skip) return;
    const int nc = w.ctrl->nc;
    if (g.npk == 1 && !rep_ran(w, nc)) return;
    int top = 0;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x)
        top = max(top, w.colour[c] + 1);
    block_atomic_max(&w.ctrl->ncolours, top);
}

static cudaError_t launch_repair(const CdGeom& g, const CdWork& w, int gc, cudaStream_t s, int* nl)
{
    cudaError_t e;
    const int gp = (g.npk + CD_BLOCK - 1) / CD_BLOCK;
    int m = (g.cap > g.n + 6) ? g.cap : g.n + 6;
    int gm = (m + CD_BLOCK - 1) / CD_BLOCK;
    if (gm > 4096) gm = 4096;
    k_rep_init<<<gp, CD_BLOCK, 0, s>>>(g, w);
    k_rep_scan_colours<<<gm, CD_BLOCK, 0, s>>>(g, w);
    k_rep_flag<<<gc, CD_BLOCK, 0, s>>>(g, w);
    *nl += 3;
    // the live contacts only (their count read on the device)
    if ((e = cd_scan_exclusive(w.rep_flag, w.rep_pos, g.cap + 1, w.scan_tmp, nullptr, s, nl, &w.ctrl->nc)) !=
        cudaSuccess)
        return e;
    k_rep_fill<<<gc, CD_BLOCK, 0, s>>>(w);
    // one warp per packing: a plain system's repair is one sequential walk
    k_rep_run<<<(g.npk + 1) / 2, 64, 0, s>>>(g, w);
    k_rep_ncolours_reset<<<1, 1, 0, s>>>(g, w);
    k_rep_ncolours<<<gc, CD_BLOCK, 0, s>>>(g, w);
    *nl += 4;
    return cudaGetLastError();
}

// Per-chunk colour histogram, layout [colour][chunk].
// Chunks of CD_CHUNK colour-order positions: only the live ones (those
// holding contacts) are counted, laid out [colour][live chunk], and scanned.
__device__ __forceinline__ int live_chunks(int nc) { return (nc + CD_CHUNK - 1) / CD_CHUNK; }

__global__ void k_chunk_hist(CdWork w)
{
    __shared__ int s_cnt[CD_KMAX];
    CdCtrl* ctrl = w.ctrl;
    if (ctrl->skip) return;
    int nc = ctrl->nc;
    const int ncl = live_chunks(nc);
    if (blockIdx.x == 0 && threadIdx.x == 0) ctrl->chunk_last = CD_KMAX * ncl - 1;
    if ((int)blockIdx.x >= ncl) return;
    for (int k = threadIdx.x; k < CD_KMAX; k += blockDim.x) s_cnt[k] = 0;
    __syncthreads();
    int c = blockIdx.x * CD_CHUNK + threadIdx.x;
    if (c < nc) {
        int k = w.colour[c];
        if (k >= 0 && k < CD_KMAX) atomicAdd(&s_cnt[k], 1);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < CD_KMAX; k += blockDim.x) w.chunk_cnt[k * ncl + blockIdx.x] = s_cnt[k];
}

template <int DIM, typename T>
__global__ void k_colour_scatter(CdGeom g, CdWork w, int pw)
{
    __shared__ int s_wcnt[CD_CHUNK / 32][CD_KMAX];
    CdCtrl* ctrl = w.ctrl;
    if (ctrl->skip) return;
    int nc = ctrl->nc;
    const int ncl = live_chunks(nc);
    if ((int)blockIdx.x >= ncl) return;
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < (CD_CHUNK / 32) * CD_KMAX; i += blockDim.x) (&s_wcnt[0][0])[i] = 0;
    __syncthreads();
    int c = blockIdx.x * CD_CHUNK + threadIdx.x;
    int k = (c < nc) ? w.colour[c] : -1;
    unsigned mask = __match_any_sync(0xffffffffu, k);
    int rank = __popc(mask & ((1u << lane) - 1u));
    if (k >= 0 && lane == __ffs(mask) - 1) s_wcnt[wid][k] = __popc(mask);
    __syncthreads();
    if (c >= nc || k < 0) return;
    for (int v = 0; v < wid; ++v) rank += s_wcnt[v][k];
    int pos = w.chunk_cnt[k * ncl + blockIdx.x] + rank;
    colour_record<DIM, T>(g, w, c, pos);
}

__global__ void k_colour_offsets(CdWork w)
{
    CdCtrl* ctrl = w.ctrl;
    if (ctrl->skip) return;
    int k = threadIdx.x;
    const int ncl = live_chunks(ctrl->nc);
    if (k < CD_KMAX) w.colour_off[k] = (ncl > 0) ? w.chunk_cnt[k * ncl] : 0;
    if (k == 0) w.colour_off[CD_KMAX] = ctrl->nc;
}

// Key-order contact range of each packing: contacts are sorted by body a and
// the packings' particles are consecutive, so packing b's contacts start at
// the first key whose a >= the packing's first particle.
__global__ void k_pk_ranges(CdGeom g, CdWork w)
{
    CdCtrl* ctrl = w.ctrl;
    if (ctrl->skip) return;
    const int nc = ctrl->nc;
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b <= g.npk; b += gridDim.x * blockDim.x) {
        if (b == g.npk) { w.pk_coff[b] = nc; continue; }
        const int first = w.pk[b].first;
        int lo = 0, hi = nc;
        while (lo < hi) {
            int mid = lo + ((hi - lo) >> 1);
            if (w.pairs[mid].x < first) lo = mid + 1; else hi = mid;
        }
        w.pk_coff[b] = lo;
    }
}

cudaError_t cd_launch_pk_ranges(const CdGeom& g, const CdWork& w, cudaStream_t s, int* nl)
{
    int gb = (g.npk + 1 + CD_BLOCK - 1) / CD_BLOCK;
    k_pk_ranges<<<gb, CD_BLOCK, 0, s>>>(g, w);
    ++*nl;
    return cudaGetLastError();
}

// Blocks per SM of the cooperative colouring grid (k_jp, and the merge's
// chain labelling, which runs on the same grid).  One keeps the grid barrier
// cheap: two made the 1e5-disc pile's colouring (29 rounds) 0.08 ms slower a
// step and the 1e6-sphere gas's (17 rounds) 0.02 ms faster.
#define CD_COLOUR_PER_SM 1

int cd_colour_max_blocks(int num_sms)
{
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_jp, CD_SWEEP_THREADS, 0) != cudaSuccess) return 0;
    const int mg = cd_merge_label_blocks_per_sm();
    if (mg > 0 && mg < per_sm) per_sm = mg;
    if (per_sm > CD_COLOUR_PER_SM) per_sm = CD_COLOUR_PER_SM;
    return per_sm * num_sms;
}

cudaError_t cd_launch_colour(const CdGeom& g, const CdWork& w, int coop_blocks, int precision, int pw,
                             cudaStream_t s, int* nl, const double* pos)
{
    cudaError_t e;
    int nchunk = (g.cap + CD_CHUNK - 1) / CD_CHUNK;
    if (nchunk < 1) nchunk = 1;
    int gc = (g.cap + CD_BLOCK - 1) / CD_BLOCK;
    if (gc < 1) gc = 1;
    if (gc > 4096) gc = 4096;
    const int nbody = g.n + (g.dyn_walls ? 6 : 0);   // particles, then force-controlled walls n + k
    if ((e = cudaMemsetAsync(w.p2c_cnt, 0, sizeof(int) * (size_t)(nbody + 1), s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(w.p2c_fill, 0, sizeof(int) * (size_t)nbody, s)) != cudaSuccess) return e;
    k_p2c_count<<<gc, CD_BLOCK, 0, s>>>(g, w); ++*nl;
    if ((e = cd_scan_exclusive(w.p2c_cnt, w.p2c_off, nbody + 1, w.scan_tmp, nullptr, s, nl)) != cudaSuccess) return e;
    k_p2c_fill<<<gc, CD_BLOCK, 0, s>>>(g, w); ++*nl;
    {
        int gn = (nbody + CD_BLOCK - 1) / CD_BLOCK;
        if (gn > 4096) gn = 4096;
        k_p2c_sort<<<gn, CD_BLOCK, 0, s>>>(g, w); ++*nl;
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (coop_blocks > 0) {
        CdGeom ga = g;
        CdWork wa = w;
        unsigned long long* prio = w.prio;
        void* args[] = {&ga, &wa, &prio};
        if ((e = cudaMemsetAsync(w.ctrl, 0, 2 * sizeof(unsigned long long), s)) != cudaSuccess) return e;
        e = cudaLaunchCooperativeKernel((const void*)k_jp, dim3(coop_blocks), dim3(CD_SWEEP_THREADS), args, 0, s);
        if (e != cudaSuccess) return e;
        ++*nl;
    }
    if ((e = launch_repair(g, w, gc, s, nl)) != cudaSuccess) return e;
    k_chunk_hist<<<nchunk, CD_CHUNK, 0, s>>>(w); ++*nl;
    if ((e = cd_scan_exclusive(w.chunk_cnt, w.chunk_cnt, CD_KMAX * nchunk, w.scan_tmp, nullptr, s, nl,
                               &w.ctrl->chunk_last)) != cudaSuccess)
        return e;
    if (g.dim == 2) {
        if (precision == CD_FP64) k_colour_scatter<2, double><<<nchunk, CD_CHUNK, 0, s>>>(g, w, pw);
        else k_colour_scatter<2, float><<<nchunk, CD_CHUNK, 0, s>>>(g, w, pw);
        ++*nl;
    } else {
        if (precision == CD_FP64) k_colour_scatter<3, double><<<nchunk, CD_CHUNK, 0, s>>>(g, w, pw);
        else k_colour_scatter<3, float><<<nchunk, CD_CHUNK, 0, s>>>(g, w, pw);
        ++*nl;
    }
    k_colour_offsets<<<1, CD_KMAX, 0, s>>>(w); ++*nl;
    return cudaGetLastError();
}
