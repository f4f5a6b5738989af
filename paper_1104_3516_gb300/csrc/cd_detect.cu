// cd_detect.cu -- contact detection with a cell list (paper Sec. 3.2) and the
// per-contact geometry (Sec. 2.1, Fig. 1; pair mass matrix of Eq. 5).
//
// Pipeline (all on one stream, sizes read from the control block so nothing
// is synchronised with the host):
//   cell_count -> scan -> cell_fill, sort    counting sort of particles by cell
//   pair_count -> scan -> capacity check     contacts per particle a (b > a)
//   pair_emit                                keys (a, b) sorted per a
//   geometry_warm -> commit                  geometry per contact, impulses carried over by key
// The pair test uses the same FP64 operation sequence as the CPU oracle
// (explicit round-to-nearest intrinsics, no FMA contraction) so the contact
// set is bit-identical to brute force.
#include "cd_detect_core.cuh"

// ---------------------------------------------------------------------------
// Exclusive scan of int32: the block sums of the tiles, then every block
// scans its tile and adds the prefix of the tiles before it.  Up to
// SCAN_FUSE tiles each block sums that prefix itself from the block sums
// (read by all blocks from L2; integer sums, so the order is immaterial);
// beyond, a single block scans the block sums in between (three passes).
// `n_dev` (device, optional) clips the scan at run time to its first
// min(*n_dev + 1, n) entries (the rest of `out` is left untouched), for
// arrays sized by capacity of which only the live contacts count.
// `total_dst` (device) receives the sum of the scanned inputs if non-null.
// In place (in == out) is allowed: a tile is read and written by the same
// threads.
// ---------------------------------------------------------------------------
#define SCAN_T 256
#define SCAN_PER 4
#define SCAN_TILE (SCAN_T * SCAN_PER)
#define SCAN_FUSE 2048

__device__ __forceinline__ int scan_extent(int n, const int* n_dev)
{
    if (!n_dev) return n;
    const int c = *n_dev + 1;
    return (c < n) ? c : n;
}

__device__ __forceinline__ int warp_incl_scan(int v)
{
    int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// Block-wide exclusive scan of one value per thread; returns the exclusive
// prefix and writes the block total to *total.
__device__ __forceinline__ int block_excl_scan(int v, int* total)
{
    __shared__ int warp_sums[SCAN_T / 32];
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int incl = warp_incl_scan(v);
    if (lane == 31) warp_sums[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        int s = (lane < SCAN_T / 32) ? warp_sums[lane] : 0;
        int si = warp_incl_scan(s);
        if (lane < SCAN_T / 32) warp_sums[lane] = si - s;
        if (lane == SCAN_T / 32 - 1) *total = si;
    }
    __syncthreads();
    int r = warp_sums[wid] + incl - v;
    __syncthreads();
    return r;
}

__global__ void k_scan_sums(const int* __restrict__ in, int n, const int* n_dev, int* __restrict__ sums)
{
    n = scan_extent(n, n_dev);
    int base = blockIdx.x * SCAN_TILE;
    if (base >= n) return;
    int s = 0;
#pragma unroll
    for (int k = 0; k < SCAN_PER; ++k) {
        int i = base + k * SCAN_T + threadIdx.x;
        if (i < n) s += in[i];
    }
    __shared__ int tot;
    block_excl_scan(s, &tot);
    if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

// Three-pass form only: one block turns the block sums into their exclusive
// prefixes.
__global__ void k_scan_top(int* sums, int n, const int* n_dev, int* total_dst)
{
    n = scan_extent(n, n_dev);
    const int nb = (n + SCAN_TILE - 1) / SCAN_TILE;
    __shared__ int carry_s;
    if (threadIdx.x == 0) carry_s = 0;
    __syncthreads();
    for (int base = 0; base < nb; base += SCAN_T) {
        int i = base + threadIdx.x;
        int v = (i < nb) ? sums[i] : 0;
        __shared__ int tot;
        int ex = block_excl_scan(v, &tot);
        int carry = carry_s;
        if (i < nb) sums[i] = carry + ex;
        __syncthreads();
        if (threadIdx.x == 0) carry_s = carry + tot;
        __syncthreads();
    }
    if (threadIdx.x == 0 && total_dst) *total_dst = carry_s;
}

// fused: the prefix of this tile from the raw block sums (else sums already
// holds the prefixes)
__global__ void k_scan_apply(const int* in, int n, const int* n_dev, const int* __restrict__ sums, int fused,
                             int* out, int* total_dst)
{
    n = scan_extent(n, n_dev);
    const int nb = (n + SCAN_TILE - 1) / SCAN_TILE;
    if ((int)blockIdx.x >= nb) return;
    __shared__ int prefix;
    if (fused) {
        int p = 0;
        for (int j = threadIdx.x; j < (int)blockIdx.x; j += SCAN_T) p += sums[j];
        block_excl_scan(p, &prefix);
    } else {
        if (threadIdx.x == 0) prefix = sums[blockIdx.x];
        __syncthreads();
    }
    int base = blockIdx.x * SCAN_TILE + threadIdx.x * SCAN_PER;
    int v[SCAN_PER];
    int s = 0;
#pragma unroll
    for (int k = 0; k < SCAN_PER; ++k) {
        int i = base + k;
        v[k] = (i < n) ? in[i] : 0;
        s += v[k];
    }
    __shared__ int tot;
    int ex = block_excl_scan(s, &tot) + prefix;
#pragma unroll
    for (int k = 0; k < SCAN_PER; ++k) {
        int i = base + k;
        if (i < n) out[i] = ex;
        ex += v[k];
    }
    if (fused && total_dst && (int)blockIdx.x == nb - 1 && threadIdx.x == 0) *total_dst = prefix + tot;
}

size_t cd_scan_tmp_ints(int n)
{
    return (size_t)((n + SCAN_TILE - 1) / SCAN_TILE + 1);
}

cudaError_t cd_scan_exclusive(const int* in, int* out, int n, int* tmp, int* total_dst, cudaStream_t stream,
                              int* nl, const int* n_dev)
{
    if (n <= 0) return cudaSuccess;
    int nb = (n + SCAN_TILE - 1) / SCAN_TILE;
    const int fused = (nb <= SCAN_FUSE || n_dev) ? 1 : 0;
    k_scan_sums<<<nb, SCAN_T, 0, stream>>>(in, n, n_dev, tmp);
    if (!fused) {
        k_scan_top<<<1, SCAN_T, 0, stream>>>(tmp, n, n_dev, total_dst);
        ++*nl;
    }
    k_scan_apply<<<nb, SCAN_T, 0, stream>>>(in, n, n_dev, tmp, fused, out, total_dst);
    *nl += 2;
    return cudaGetLastError();
}

template <int DIM>
__global__ void k_cell_count(CdGeom g, CdWork w, const double* __restrict__ pos, const double* __restrict__ radius,
                             int* __restrict__ cell_of, int* __restrict__ cell_cnt, const CdCtrl* ctrl)
{
    if (ctrl->skip) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.n; i += gridDim.x * blockDim.x)
        count_cell<DIM>(g, w, pos, radius, i, cell_of, cell_cnt);
}

__global__ void k_cell_fill(int n, const int* __restrict__ cell_of, const int* __restrict__ cell_start,
                            int* __restrict__ cell_fill, int* __restrict__ cell_pid, const CdCtrl* ctrl)
{
    if (ctrl->skip) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        int c = cell_of[i];
        int slot = atomicAdd(&cell_fill[c], 1);
        cell_pid[cell_start[c] + slot] = i;
    }
}

// Each cell's particle list in ascending id order (the atomic fill leaves it
// in arrival order): lets the pair walk skip a whole cell whose last id is
// not above the particle's own.
__global__ void k_cell_sort(int ncell, const int* __restrict__ cell_start, int* __restrict__ cell_pid,
                            const CdCtrl* ctrl)
{
    if (ctrl->skip) return;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ncell; c += gridDim.x * blockDim.x) {
        const int b = cell_start[c], e = cell_start[c + 1];
        for (int k = b + 1; k < e; ++k) {
            const int v = cell_pid[k];
            int j = k - 1;
            while (j >= b && cell_pid[j] > v) { cell_pid[j + 1] = cell_pid[j]; --j; }
            cell_pid[j + 1] = v;
        }
    }
}

template <int DIM>
__global__ void __launch_bounds__(CD_BLOCK, 4)
k_pair_count(CdGeom g, CdWork w, const double* __restrict__ pos, const double* __restrict__ radius,
                             const int* __restrict__ cell_of, const int* __restrict__ cell_start,
                             const int* __restrict__ cell_pid, int* __restrict__ pcnt, CdCtrl* ctrl)
{
    __shared__ int s_qb[CD_BLOCK / 32][CD_QUEUE], s_qo[CD_BLOCK / 32][CD_QUEUE];
    __shared__ int s_cnt[CD_BLOCK];
    __shared__ int s_lo[Runs<DIM>::N][CD_BLOCK], s_hi[Runs<DIM>::N][CD_BLOCK];
    if (ctrl->skip) return;
    const int wq = threadIdx.x >> 5;
    // warps step through the particles together (the loop bound is warp-uniform)
    for (int base = blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < g.n; base += gridDim.x * blockDim.x)
        count_pairs<DIM, CD_BLOCK, true>(g, w, pos, radius, base, g.n, cell_of, cell_start, cell_pid, pcnt, s_qb[wq],
                                         s_qo[wq], s_cnt + 32 * wq, &s_lo[0][0], &s_hi[0][0]);
}

// Capacity check after the scan of the per-particle counts.
__global__ void k_cap_check(CdCtrl* ctrl, int cap)
{
    if (ctrl->skip) return;
    if (ctrl->nc_needed > cap || ctrl->error != CDE_NONE) {
        ctrl->overflow = (ctrl->nc_needed > cap) ? 1 : ctrl->overflow;
        ctrl->skip = 1;
    }
}

template <int DIM>
__device__ __forceinline__ void store_geometry(const CdWork& w, int c, int a, int b, const double nv[3], double gap,
                                               double mn, double mt)
{
    w.pairs_nx[c] = make_int2(a, b);
    w.nrm[3 * c + 0] = nv[0];
    w.nrm[3 * c + 1] = nv[1];
    w.nrm[3 * c + 2] = nv[2];
    w.gap[c] = gap;
    w.mn[c] = mn;
    w.mt[c] = mt;
}

template <int DIM>
__global__ void k_pair_emit(CdGeom g, CdWork w, const double* __restrict__ pos, const double* __restrict__ radius)
{
    if (w.ctrl->skip) return;
    for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < g.n; a += gridDim.x * blockDim.x)
        emit_pairs<DIM, true>(g, w, pos, radius, a, w.poff[a], w.cell_start);
}

template <int DIM>
__global__ void k_geometry_warm(CdGeom g, CdWork w, const double* __restrict__ pos, const double* __restrict__ radius,
                                const double* __restrict__ inv_m, const double* __restrict__ inv_I, int warm, int pw)
{
    CdCtrl* ctrl = w.ctrl;
    if (ctrl->skip) return;
    const int nnew = ctrl->nc_needed;
    const int nold = ctrl->nc;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nnew; c += gridDim.x * blockDim.x)
        geometry_warm<DIM>(g, w, c, nold, ctrl->prev_offsets, pos, radius, inv_m, inv_I, warm, pw);
}

// Geometry of a caller-supplied contact list (already in pairs_nx).
template <int DIM>
__global__ void k_geometry_given(CdGeom g, CdWork w, int nc, const double* __restrict__ pos,
                                 const double* __restrict__ radius, const double* __restrict__ inv_m,
                                 const double* __restrict__ inv_I)
{
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x) {
        int2 ab = w.pairs_nx[c];
        double nv[3], gap, mn, mt;
        contact_geometry<DIM>(g, w, ab.x, ab.y, pos, radius, inv_m, inv_I, nv, &gap, &mn, &mt);
        store_geometry<DIM>(w, c, ab.x, ab.y, nv, gap, mn, mt);
    }
}

__global__ void k_copy_pairs(int nc, const int32_t* __restrict__ src, int2* __restrict__ dst, CdCtrl* ctrl)
{
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x)
        dst[c] = make_int2(src[2 * c], src[2 * c + 1]);
    if (blockIdx.x == 0 && threadIdx.x == 0) ctrl->nc_needed = nc;
}

// Caller-given starting impulses (or zeros) for a caller-given list.
__global__ void k_given_impulses(CdWork w, int nc, const double* __restrict__ imp, int pw)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nc * pw; i += gridDim.x * blockDim.x)
        w.Pk_nx[i] = imp ? imp[i] : 0.0;
}

// The new set becomes the current one; with `n` > 0 (a detected set) the
// per-particle offsets of the detection are kept for the next warm start.
__global__ void k_commit(CdWork w, int pw, int n)
{
    CdCtrl* ctrl = w.ctrl;
    if (ctrl->skip) return;
    int nc = ctrl->nc_needed;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x) {
        w.pairs[c] = w.pairs_nx[c];
        for (int k = 0; k < pw; ++k) w.Pk[pw * c + k] = w.Pk_nx[pw * c + k];
    }
    if (w.poff_prev && n > 0)
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n + 1; i += gridDim.x * blockDim.x)
            w.poff_prev[i] = w.poff[i];
}

// by_particle: the new set's per-particle offsets are in poff_prev.
__global__ void k_set_nc(CdCtrl* ctrl, int by_particle)
{
    if (ctrl->skip) return;
    ctrl->nc = ctrl->nc_needed;
    ctrl->prev_offsets = by_particle;
    ctrl->order_nc = -1;
    ctrl->order_lost = 0;
}

static int grid_for(int n, int per_block = CD_BLOCK)
{
    int g = (n + per_block - 1) / per_block;
    if (g < 1) g = 1;
    if (g > 4096) g = 4096;
    return g;
}

cudaError_t cd_launch_detect(const CdGeom& g, const CdWork& w, const double* pos, const double* radius,
                             const double* inv_m, const double* inv_I, int warm, int pw, cudaStream_t s, int* nl)
{
    int ncell = g.ncell_total;
    cudaError_t e;
    if ((e = cudaMemsetAsync(w.cell_cnt, 0, sizeof(int) * (size_t)(ncell + 1), s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(w.cell_fill, 0, sizeof(int) * (size_t)ncell, s)) != cudaSuccess) return e;
    int gb = grid_for(g.n);
    if (g.dim == 2) k_cell_count<2><<<gb, CD_BLOCK, 0, s>>>(g, w, pos, radius, w.cell_of, w.cell_cnt, w.ctrl);
    else k_cell_count<3><<<gb, CD_BLOCK, 0, s>>>(g, w, pos, radius, w.cell_of, w.cell_cnt, w.ctrl);
    ++*nl;
    if ((e = cd_scan_exclusive(w.cell_cnt, w.cell_start, ncell + 1, w.scan_tmp, nullptr, s, nl)) != cudaSuccess) return e;
    k_cell_fill<<<gb, CD_BLOCK, 0, s>>>(g.n, w.cell_of, w.cell_start, w.cell_fill, w.cell_pid, w.ctrl); ++*nl;
    k_cell_sort<<<grid_for(ncell), CD_BLOCK, 0, s>>>(ncell, w.cell_start, w.cell_pid, w.ctrl); ++*nl;
    if (g.dim == 2)
        k_pair_count<2><<<gb, CD_BLOCK, 0, s>>>(g, w, pos, radius, w.cell_of, w.cell_start, w.cell_pid, w.pcnt,
                                                w.ctrl);
    else
        k_pair_count<3><<<gb, CD_BLOCK, 0, s>>>(g, w, pos, radius, w.cell_of, w.cell_start, w.cell_pid, w.pcnt,
                                                w.ctrl);
    ++*nl;
    if ((e = cudaMemsetAsync(w.pcnt + g.n, 0, sizeof(int), s)) != cudaSuccess) return e;
    if ((e = cd_scan_exclusive(w.pcnt, w.poff, g.n + 1, w.scan_tmp, &w.ctrl->nc_needed, s, nl)) != cudaSuccess) return e;
    k_cap_check<<<1, 1, 0, s>>>(w.ctrl, g.cap); ++*nl;
    if (g.dim == 2) k_pair_emit<2><<<gb, CD_BLOCK, 0, s>>>(g, w, pos, radius);
    else k_pair_emit<3><<<gb, CD_BLOCK, 0, s>>>(g, w, pos, radius);
    ++*nl;
    int gc = grid_for(g.cap);
    if (g.dim == 2) k_geometry_warm<2><<<gc, CD_BLOCK, 0, s>>>(g, w, pos, radius, inv_m, inv_I, warm, pw);
    else k_geometry_warm<3><<<gc, CD_BLOCK, 0, s>>>(g, w, pos, radius, inv_m, inv_I, warm, pw);
    ++*nl;
    k_commit<<<gc, CD_BLOCK, 0, s>>>(w, pw, g.n); ++*nl;
    k_set_nc<<<1, 1, 0, s>>>(w.ctrl, w.poff_prev != nullptr); ++*nl;
    return cudaGetLastError();
}

cudaError_t cd_launch_set_contacts(const CdGeom& g, const CdWork& w, const double* pos, const double* radius,
                                   const double* inv_m, const double* inv_I, int nc, const int32_t* pairs,
                                   const double* impulses, int pw, cudaStream_t s, int* nl)
{
    int gc = grid_for(nc > 0 ? nc : 1);
    k_copy_pairs<<<gc, CD_BLOCK, 0, s>>>(nc, pairs, w.pairs_nx, w.ctrl); ++*nl;
    if (nc > 0) {
        if (g.dim == 2) k_geometry_given<2><<<gc, CD_BLOCK, 0, s>>>(g, w, nc, pos, radius, inv_m, inv_I);
        else k_geometry_given<3><<<gc, CD_BLOCK, 0, s>>>(g, w, nc, pos, radius, inv_m, inv_I);
        ++*nl;
    }
    k_given_impulses<<<grid_for(nc * pw > 0 ? nc * pw : 1), CD_BLOCK, 0, s>>>(w, nc, impulses, pw); ++*nl;
    k_commit<<<gc, CD_BLOCK, 0, s>>>(w, pw, 0); ++*nl;   // a caller-given list: no offsets
    k_set_nc<<<1, 1, 0, s>>>(w.ctrl, 0); ++*nl;
    return cudaGetLastError();
}
