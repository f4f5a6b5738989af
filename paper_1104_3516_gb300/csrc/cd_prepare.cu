// cd_prepare.cu -- detection, colouring, colour ordering and the free-flight
// velocities of a plain system in one kernel.
//
// The stages are those of cd_detect.cu and cd_colour.cu, about fifteen with a
// barrier of the blocks between them in place of ~45 launches (2 to 4 us each
// on a small system, whatever they do).  What is left is latency: a stage is
// two to eight dependent trips to L2 (300 to 650 cycles each, the L1 being
// empty after every barrier) and a barrier.  So stages are merged where the
// data allow: scans are finished by their readers (each block scans its chunk,
// the sums of the chunks before come from shared memory); a block counts,
// writes and measures the contacts of its own particles; a body's own contacts
// are a range of the key order and only those in which it is body b are
// gathered and sorted; cell lists stay unsorted.
//
// Step of a 1,000-disc rollout 180 -> 101 us (of it this kernel 57 us; 84 us with
// the shorter solve since), 10,000 discs 175 -> 127, detection without workspace
// 151 -> 112 us (90 with the grid laid out on the device).  The largest size that takes it: 3D step (150,000 / 400,000 / 1,000,000
// spheres) 393 -> 336, 1,018 -> 1,003, 2,319 -> 2,378 us: the walks of a
// million spheres want the occupancy of kernels of their own.
#include "cd_colour_core.cuh"
#include "cd_detect_core.cuh"
#include "cd_pack_core.cuh"

#define PREP_THREADS 512
#define PREP_WARPS (PREP_THREADS / 32)
#define PREP_CLUSTER 16
enum { PREP_CELLS = 0, PREP_CONTACTS, PREP_P2C, PREP_DEGREE };   // per-block values in prep_tot

// The barrier of the kernel's blocks: of their cluster, or of the grid.
struct PrepSync {
    CdCtrl* ctrl;
    unsigned long long epoch;
    int cluster;
    __device__ __forceinline__ bool operator()()
    {
        if (cluster) {
            asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
            return true;
        }
        return cd_grid_sync(ctrl, gridDim.x, epoch);
    }
};

// Exclusive prefixes that are complete within each block's chunk (2^shift
// entries, in order) only, with the sums of the chunks before beside them.
struct PrepPrefix {
    const int* local;
    const int* before;
    int shift;
    __device__ __forceinline__ int operator[](int i) const { return local[i] + before[i >> shift]; }
};

// Shared memory of a block.
struct PrepShared {
    int cells[CD_PREP_MAX_BLOCKS], p2c[CD_PREP_MAX_BLOCKS];   // sums of the chunks before each block's
    int warp[PREP_WARPS];
    int total;
    int hist[CD_KMAX];                                  // contacts per colour, then the next position of each
    int wcnt[PREP_WARPS][CD_KMAX];
    int coff[CD_KMAX + 1];
    int top, dmax;
};

// Exclusive scan of in[lo .. hi) into out (may be in), the block together;
// returns the sum in every thread.
__device__ __forceinline__ int prep_scan(const int* in, int* out, int lo, int hi, PrepShared& sh)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int run = 0;
    for (int i0 = lo; i0 < hi; i0 += PREP_THREADS) {
        const int i = i0 + (int)threadIdx.x;
        const int v = (i < hi) ? in[i] : 0;
        int incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) sh.warp[wid] = incl;
        __syncthreads();
        int before = 0, tile = 0;
#pragma unroll
        for (int q = 0; q < PREP_WARPS; ++q) {
            const int c = sh.warp[q];
            if (q < wid) before += c;
            tile += c;
        }
        if (i < hi) out[i] = run + before + incl - v;
        run += tile;
        __syncthreads();
    }
    return run;
}

// Sums of the values of the blocks before each block, into dst (shared); the
// sum of all in every thread.  One warp works.
__device__ __forceinline__ int prep_before(const int* tot, int nb, int* dst, PrepShared& sh)
{
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        int run = 0;
        for (int b0 = 0; b0 < nb; b0 += 32) {
            const int b = b0 + lane;
            const int v = (b < nb) ? tot[b] : 0;
            int incl = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            if (b < nb) dst[b] = run + incl - v;
            run += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (lane == 0) sh.total = run;
    }
    __syncthreads();
    const int r = sh.total;
    __syncthreads();
    return r;
}

__host__ __device__ __forceinline__ int prep_shift(int count, int nb)
{
    int s = 5;
    while (((long long)nb << s) < count) ++s;
    return s;
}

// False when a barrier gave up: the step must not go on.
template <int DIM, typename T, bool DETECT_ONLY>
__device__ __forceinline__ bool prepare(const CdGeom& g, const CdWork& w, const CdPrepIO& io, int cluster, int* s_dyn,
                                        PrepShared& sh)
{
    CdCtrl* ctrl = w.ctrl;
    const int nb = gridDim.x, blk = blockIdx.x;
    const int tid = blk * PREP_THREADS + (int)threadIdx.x, stride = nb * PREP_THREADS;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int n = g.n, ncell = g.ncell_total;
    const int nbody = n + (g.dyn_walls ? 6 : 0);
    const int nold = ctrl->nc, by_particle = ctrl->prev_offsets;
    PrepSync sync{ctrl, 0ULL, cluster};
    int* tot = w.prep_tot;
    // this block's chunks: cells (and the end), bodies (and the end), particles
    const int cshift = prep_shift(ncell + 1, nb), bshift = prep_shift(nbody + 1, nb);
    const int cell0 = min(blk << cshift, ncell + 1), cell1 = min((blk + 1) << cshift, ncell + 1);
    const int body0 = min(blk << bshift, nbody + 1), body1 = min((blk + 1) << bshift, nbody + 1);
    const int per = ((n + nb - 1) / nb + 31) & ~31;
    const int part0 = min(blk * per, n), part1 = min(part0 + per, n);

    for (int i = tid; i <= ncell; i += stride) {
        w.cell_cnt[i] = 0;
        if (i < ncell) w.cell_fill[i] = 0;
    }
    if (!DETECT_ONLY) {
        for (int i = tid; i <= nbody; i += stride) {
            w.p2c_cnt[i] = 0;
            if (i < nbody) w.p2c_fill[i] = 0;
        }
    }
    if (!sync()) return false;

    // cell lists (in no order)
    for (int i = tid; i < n; i += stride) count_cell<DIM>(g, w, io.pos, io.radius, i, w.cell_of, w.cell_cnt);
    if (!DETECT_ONLY && io.pack)
        pack_velocities<DIM, T>(g, w, io.vel, io.omega, io.inv_m, io.f_ext, io.free_flight, tid, stride, blk == 0);
    if (!sync()) return false;
    {
        const int t = prep_scan(w.cell_cnt, w.cell_start, cell0, cell1, sh);
        if (threadIdx.x == 0) tot[PREP_CELLS * nb + blk] = t;
    }
    if (!sync()) return false;
    prep_before(tot + PREP_CELLS * nb, nb, sh.cells, sh);
    const PrepPrefix start{w.cell_start, sh.cells, cshift};
    for (int i = tid; i < n; i += stride) {
        const int c = w.cell_of[i];
        w.cell_pid[start[c] + atomicAdd(&w.cell_fill[c], 1)] = i;
    }
    if (!sync()) return false;

    // contacts of the block's particles: counted, then written from the sum
    // of the blocks before on
    {
        int* const qb = s_dyn + CD_QUEUE * wid;
        int* const qo = s_dyn + CD_QUEUE * (PREP_WARPS + wid);
        int* const cnt = s_dyn + 2 * CD_QUEUE * PREP_WARPS + 32 * wid;
        int* const runs = s_dyn + 2 * CD_QUEUE * PREP_WARPS + PREP_THREADS;
        for (int base = part0 + 32 * wid; base < part1; base += PREP_THREADS)
            count_pairs<DIM, PREP_THREADS, false>(g, w, io.pos, io.radius, base, part1, w.cell_of, start, w.cell_pid,
                                                  w.pcnt, qb, qo, cnt, runs, runs + Runs<DIM>::N * PREP_THREADS);
        __syncthreads();
        const int t = prep_scan(w.pcnt, w.poff, part0, part1, sh);
        if (threadIdx.x == 0) tot[PREP_CONTACTS * nb + blk] = t;
    }
    if (!sync()) return false;
    const int nc = prep_before(tot + PREP_CONTACTS * nb, nb, sh.p2c, sh);
    const int c0 = sh.p2c[blk], c1 = c0 + tot[PREP_CONTACTS * nb + blk];
    const bool fits = nc <= g.cap && cd_ld_volatile_int(&ctrl->error) == CDE_NONE;
    if (tid == 0) {
        ctrl->nc_needed = nc;
        if (!fits) {
            if (nc > g.cap) ctrl->overflow = 1;
            ctrl->skip = 1;
        }
    }
    if (!fits) return true;
    for (int a = part0 + (int)threadIdx.x; a < part1; a += PREP_THREADS) {
        const int o = w.poff[a] + c0;
        w.poff[a] = o;
        emit_pairs<DIM, false>(g, w, io.pos, io.radius, a, o, start);
        if (!DETECT_ONLY) atomicAdd(&w.p2c_cnt[a], w.pcnt[a]);
    }
    if (blk == nb - 1 && threadIdx.x == 0) w.poff[n] = nc;
    __syncthreads();
    for (int c = c0 + (int)threadIdx.x; c < c1; c += PREP_THREADS) {
        geometry_warm<DIM>(g, w, c, nold, by_particle, io.pos, io.radius, io.inv_m, io.inv_I, io.warm, io.pw);
        const int b = w.pairs_nx[c].y;
        if (!DETECT_ONLY && cd_is_body(g, b)) atomicAdd(&w.p2c_cnt[b], 1);
    }
    if (!sync()) return false;

    // the new set becomes the current one
    for (int c = c0 + (int)threadIdx.x; c < c1; c += PREP_THREADS) {
        w.pairs[c] = w.pairs_nx[c];
        for (int k = 0; k < io.pw; ++k) w.Pk[io.pw * c + k] = w.Pk_nx[io.pw * c + k];
    }
    if (w.poff_prev) {
        for (int a = part0 + (int)threadIdx.x; a < part1; a += PREP_THREADS) w.poff_prev[a] = w.poff[a];
        if (blk == nb - 1 && threadIdx.x == 0) w.poff_prev[n] = nc;
    }
    if (tid == 0) {
        ctrl->nc = nc;
        ctrl->prev_offsets = (w.poff_prev != nullptr);
        ctrl->order_nc = -1;
        ctrl->order_lost = 0;
    }
    if (DETECT_ONLY) return true;

    // contacts of each body in ascending order: those in which it is body b,
    // then its own
    {
        const int t = prep_scan(w.p2c_cnt, w.p2c_cnt, body0, body1, sh);
        if (threadIdx.x == 0) tot[PREP_P2C * nb + blk] = t;
    }
    if (!sync()) return false;
    prep_before(tot + PREP_P2C * nb, nb, sh.p2c, sh);
    const PrepPrefix first{w.p2c_cnt, sh.p2c, bshift};
    for (int i = body0 + (int)threadIdx.x; i < body1; i += PREP_THREADS) w.p2c_off[i] = first[i];
    for (int c = c0 + (int)threadIdx.x; c < c1; c += PREP_THREADS) {
        const int2 ab = w.pairs[c];
        w.p2c[first[ab.x + 1] - (w.poff[ab.x + 1] - c)] = c;
        if (cd_is_body(g, ab.y)) w.p2c[first[ab.y] + atomicAdd(&w.p2c_fill[ab.y], 1)] = c;
    }
    if (!sync()) return false;
    for (int i = tid; i < nbody; i += stride) {
        const int b = w.p2c_off[i], e = w.p2c_off[i + 1] - ((i < n) ? w.poff[i + 1] - w.poff[i] : 0);
        for (int k = b + 1; k < e; ++k) {
            const int v = w.p2c[k];
            int j = k - 1;
            while (j >= b && w.p2c[j] > v) { w.p2c[j + 1] = w.p2c[j]; --j; }
            w.p2c[j + 1] = v;
        }
    }
    if (!jp_colour(g, w, nc, w.prio, sync)) return false;
    if (cd_ld_volatile_int(&ctrl->error) != CDE_NONE) {
        if (tid == 0) ctrl->skip = 1;
        return true;
    }

    // colours of the block's contacts, and whether the highest one is repaired
    const int K = cd_ld_volatile_int(&ctrl->ncolours);   // (the repair may take some away)
    for (int round = 0; round < 2; ++round) {
        for (int k = threadIdx.x; k < CD_KMAX; k += PREP_THREADS) sh.hist[k] = 0;
        if (threadIdx.x == 0) sh.dmax = 0;
        __syncthreads();
        for (int c = c0 + (int)threadIdx.x; c < c1; c += PREP_THREADS) atomicAdd(&sh.hist[w.colour[c]], 1);
        if (round == 0) {
            int d = 0;
            for (int i = tid; i < nbody; i += stride)
                d = max(d, w.p2c_off[i + 1] - w.p2c_off[i]);
            d = __reduce_max_sync(0xffffffffu, d);
            if (lane == 0) atomicMax(&sh.dmax, d);
        }
        __syncthreads();
        for (int k = threadIdx.x; k < CD_KMAX; k += PREP_THREADS) w.prep_hist[k * nb + blk] = sh.hist[k];
        if (round == 0 && threadIdx.x == 0) tot[PREP_DEGREE * nb + blk] = sh.dmax;
        if (!sync()) return false;
        if (round == 1) break;
        if (wid == 0) {
            int top = 0, before = 0, dmax = 0;
            for (int b = lane; b < nb; b += 32) {
                const int v = (K > 0) ? w.prep_hist[(K - 1) * nb + b] : 0;
                top += v;
                if (b < blk) before += v;
                dmax = max(dmax, tot[PREP_DEGREE * nb + b]);
            }
            top = __reduce_add_sync(0xffffffffu, top);
            before = __reduce_add_sync(0xffffffffu, before);
            dmax = __reduce_max_sync(0xffffffffu, dmax);
            if (lane == 0) { sh.top = top; sh.total = before; sh.dmax = dmax; }
        }
        __syncthreads();
        if (!rep_wanted(nc, K - 1, sh.dmax, sh.top)) break;
        // the contacts of the highest colour in key order, each block its own; then
        // the repair by one warp.  (Listed by one block, as they were, and the colours
        // counted anew by it, 400,000 packed discs' 894,000 contacts took it 0.8 ms.)
        if (sh.hist[K - 1] > 0) {
            int run = sh.total;
            for (int i0 = c0; i0 < c1; i0 += PREP_THREADS) {
                const int c = i0 + (int)threadIdx.x;
                const bool f = c < c1 && w.colour[c] == K - 1;
                const unsigned m = __ballot_sync(0xffffffffu, f);
                if (lane == 0) sh.warp[wid] = __popc(m);
                __syncthreads();
                int at = run;
                for (int q = 0; q < PREP_WARPS; ++q) {
                    if (q < wid) at += sh.warp[q];
                    run += sh.warp[q];
                }
                if (f) w.rep_list[at + __popc(m & ((1u << lane) - 1u))] = c;
                __syncthreads();
            }
        }
        if (!sync()) return false;
        if (blk == 0 && wid == 0) rep_run(g, w, K - 1, 0, sh.top, nc, w.rep_path);
        if (!sync()) return false;
    }

    // stable partition by colour: where each colour starts, and where this
    // block's contacts of it do
    for (int k = wid; k < CD_KMAX; k += PREP_WARPS) {
        int all = 0, mine = 0;
        if (k < K) {
            for (int b = lane; b < nb; b += 32) {
                const int v = w.prep_hist[k * nb + b];
                all += v;
                if (b < blk) mine += v;
            }
            all = __reduce_add_sync(0xffffffffu, all);
            mine = __reduce_add_sync(0xffffffffu, mine);
        }
        if (lane == 0) { sh.coff[k] = all; sh.hist[k] = mine; }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int run = 0, top = 0;
        for (int k = 0; k < CD_KMAX; ++k) {
            const int v = sh.coff[k];
            sh.coff[k] = run;
            sh.hist[k] += run;
            run += v;
            if (v > 0) top = k + 1;
        }
        sh.coff[CD_KMAX] = nc;
        if (blk == 0) ctrl->ncolours = top;
    }
    __syncthreads();
    if (blk == 0)
        for (int k = threadIdx.x; k <= CD_KMAX; k += PREP_THREADS) w.colour_off[k] = sh.coff[k];
    if (tid == 0) ctrl->order_nc = nc;   // (no barrier follows; a block that gave up at the last one has set order_lost)
    for (int i0 = c0; i0 < c1; i0 += PREP_THREADS) {
        for (int i = threadIdx.x; i < PREP_WARPS * CD_KMAX; i += PREP_THREADS) (&sh.wcnt[0][0])[i] = 0;
        __syncthreads();
        const int c = i0 + (int)threadIdx.x;
        const int k = (c < c1) ? w.colour[c] : -1;
        const unsigned m = __match_any_sync(0xffffffffu, k);
        int rank = __popc(m & ((1u << lane) - 1u));
        if (k >= 0 && lane == __ffs(m) - 1) sh.wcnt[wid][k] = __popc(m);
        __syncthreads();
        if (k >= 0) {
            for (int q = 0; q < wid; ++q) rank += sh.wcnt[q][k];
            colour_record<DIM, T>(g, w, c, sh.hist[k] + rank);
        }
        __syncthreads();
        for (int q = threadIdx.x; q < CD_KMAX; q += PREP_THREADS) {
            int t = 0;
            for (int u = 0; u < PREP_WARPS; ++u) t += sh.wcnt[u][q];
            sh.hist[q] += t;
        }
        __syncthreads();
    }
    return true;
}

template <int DIM, typename T>
__global__ void __launch_bounds__(PREP_THREADS, 1) k_prepare(CdGeom g, CdWork w, CdPrepIO io, int cluster)
{
    extern __shared__ int s_dyn[];   // the counting pass's queues and runs
    __shared__ PrepShared sh;
    if (w.ctrl->skip) return;
    const bool ok = prepare<DIM, T, false>(g, w, io, cluster, s_dyn, sh);
    if (threadIdx.x == 0 && !ok) {   // (any block that gave up says so: the one that reports the errors may have left first)
        w.ctrl->skip = 1;
        w.ctrl->order_lost = 1;
    }
}

// The contact set alone, on a grid that the device laid out.
template <int DIM>
__global__ void __launch_bounds__(PREP_THREADS, 1) k_detect(CdGeom given, CdWork w, CdPrepIO io, int cluster)
{
    extern __shared__ int s_dyn[];
    __shared__ PrepShared sh;
    __shared__ CdGeom g;   // (a changed copy in registers would go to local memory)
    if (w.ctrl->skip || io.grid->status != CDG_OK) return;
    if (threadIdx.x == 0) g = given;
    __syncthreads();
    if (threadIdx.x < 3) {
        g.cs[threadIdx.x] = io.grid->cs[threadIdx.x];
        g.inv_cs[threadIdx.x] = io.grid->inv_cs[threadIdx.x];
        g.ncell[threadIdx.x] = io.grid->ncell[threadIdx.x];
    }
    if (threadIdx.x == 3) g.ncell_total = io.grid->total;
    __syncthreads();
    if (!prepare<DIM, double, true>(g, w, io, cluster, s_dyn, sh) && threadIdx.x == 0) w.ctrl->skip = 1;
}

static const void* prep_fn(int dim, int precision, int detect_only)
{
    if (detect_only) return dim == 2 ? (const void*)k_detect<2> : (const void*)k_detect<3>;
    if (dim == 2) return precision == CD_FP64 ? (const void*)k_prepare<2, double> : (const void*)k_prepare<2, float>;
    return precision == CD_FP64 ? (const void*)k_prepare<3, double> : (const void*)k_prepare<3, float>;
}

static size_t prep_shared_bytes(int dim)
{
    const int runs = (dim == 3) ? Runs<3>::N : Runs<2>::N;
    return sizeof(int) * (size_t)(2 * CD_QUEUE * PREP_WARPS + PREP_THREADS + 2 * runs * PREP_THREADS);
}

static cudaLaunchConfig_t prep_config(int dim, int blocks, int cluster, cudaLaunchAttribute* a)
{
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(blocks);
    c.blockDim = dim3(PREP_THREADS);
    c.dynamicSmemBytes = prep_shared_bytes(dim);
    c.attrs = a;
    c.numAttrs = 1;
    if (cluster) {
        a->id = cudaLaunchAttributeClusterDimension;
        a->val.clusterDim.x = (unsigned)blocks;
        a->val.clusterDim.y = a->val.clusterDim.z = 1;
    } else {
        a->id = cudaLaunchAttributeCooperative;
        a->val.cooperative = 1;
    }
    return c;
}

// One cluster of 16 blocks for small systems, whose barrier is cheaper (0.5 to
// 0.85 us against 1.4 us), the whole grid for larger ones, whose FP64 work
// (geometry) and walks want all SMs.  Rollout step, cluster / grid / separate
// kernels: 2D 1,000 discs 105 / 115 / 155 us, 5,000 111 / 118 / 165, 10,000
// 129 / 127 / 175, 40,000 185 / 144 / 191; 3D 1,000 spheres 162 / 169 / 222,
// 5,000 188 / 192 / 242, 20,000 307 / 205 / 261, 50,000 544 / 228 / 290.
//
// Few particles in a large box: the cells are cleared and scanned all the same,
// by 16 SMs 512 a block at a time, or by all, against separate kernels that scan
// 2,048 a block.  Steps of 1,000 discs in a box of 1e5 cells 95 / 94 / 217 us, 3e5 120
// / 95 / 219, 1e6 159 / 103 / 219, 4e6 377 / 135 / 240, 1e7 1,623 / - / 219; 500,000
// discs in 4e6 cells - / 463 / 485, 5e6 - / 519 / 490, 1e7 - / 646 / 541 (the chunks
// of cells are powers of two: beyond 152 x 2^15 half the blocks have none).
#define PREP_CLUSTER_CELLS (1 << 17)
#define PREP_MAX_CELLS (1 << 22)
int cd_prepare_cluster_n(int dim) { return dim == 2 ? 7000 : 5000; }

CdPrepPlan cd_prepare_plan(int dim, int precision, int detect_only, int64_t n, int64_t cells, int device)
{
    CdPrepPlan plan = {0, 0};
    if (n > CD_PREP_MAX_N || cells > PREP_MAX_CELLS) return plan;
    const void* f = prep_fn(dim, precision, detect_only);
    const size_t bytes = prep_shared_bytes(dim);
    cudaLaunchAttribute a[1];
    int b = 0, sms = 0;
    if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess) return plan;
    if (n <= cd_prepare_cluster_n(dim) && cells <= PREP_CLUSTER_CELLS &&
        cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
        const cudaLaunchConfig_t c = prep_config(dim, PREP_CLUSTER, 1, a);
        if (cudaOccupancyMaxActiveClusters(&b, f, &c) == cudaSuccess && b >= 1) return {PREP_CLUSTER, 1};
    }
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return plan;
    if (sms > CD_PREP_MAX_BLOCKS) sms = CD_PREP_MAX_BLOCKS;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, f, PREP_THREADS, bytes) == cudaSuccess && b >= 1)
        plan.blocks = sms;
    return plan;
}

cudaError_t cd_launch_prepare(const CdGeom& g, const CdWork& w, const CdPrepIO& io, int blocks, int cluster,
                              int precision, cudaStream_t s, int* nl)
{
    CdGeom ga = g;
    CdWork wa = w;
    CdPrepIO ia = io;
    int cl = cluster;
    void* args[] = {&ga, &wa, &ia, &cl};
    if (!cluster) {
        cudaError_t e = cudaMemsetAsync(w.ctrl, 0, 2 * sizeof(unsigned long long), s);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchAttribute a[1];
    cudaLaunchConfig_t c = prep_config(g.dim, blocks, cluster, a);
    c.stream = s;
    ++*nl;
    return cudaLaunchKernelExC(&c, prep_fn(g.dim, precision, io.grid != nullptr), args);
}
