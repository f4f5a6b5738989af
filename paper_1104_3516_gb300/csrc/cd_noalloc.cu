// cd_noalloc.cu -- contact detection for callers that cannot allocate device
// memory.
//
// Some hosts of this library run where cudaMalloc is not available to them:
// code inside a framework that owns every device allocation, a plug-in that
// may only use buffers handed to it, or a caller that must not allocate while
// a memory budget is fixed.  cd_detect_contacts_noalloc gives them the cell-
// list detection of cd_detect_contacts without a system object or workspace:
// its scratch (cell grid, per-particle counts and offsets, scan temporaries,
// pair mass matrix, a control block) lives in the file-scope device array
// below, which every GPU that loads the library holds until the process
// exits.
//
// The host cannot use the array's name as a device address, so on the first
// call on each device (with that device current) the address is looked up
// once with cudaGetSymbolAddress and cached; that first call therefore must
// not happen during stream capture.  All calls share the array and it keeps
// the last call's contents: every call clears what must start at zero, and
// calls that overlap on the GPU (two streams, two threads) race on it.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>

#include "cd_internal.cuh"

#define CD_NOALLOC_MAX_N 16384
#define CD_NOALLOC_MAX_CELLS 65536
#define CD_NOALLOC_MAX_CONTACTS 65536
#define CD_NOALLOC_MAX_DEVICES 64

// Byte layout of the scratch (each part 256-byte aligned).
#define NA_ALIGN(x) ((((size_t)(x)) + 255) & ~(size_t)255)
#define NA_CTRL 0
#define NA_I32(count) NA_ALIGN(sizeof(int) * (size_t)(count))
#define NA_GRID (NA_CTRL + NA_ALIGN(sizeof(CdCtrl)))   // (read back with the control block)
#define NA_CELL_OF (NA_GRID + NA_ALIGN(sizeof(CdGridSpec)))
#define NA_CELL_CNT (NA_CELL_OF + NA_I32(CD_NOALLOC_MAX_N))
#define NA_CELL_START (NA_CELL_CNT + NA_I32(CD_NOALLOC_MAX_CELLS + 1))
#define NA_CELL_FILL (NA_CELL_START + NA_I32(CD_NOALLOC_MAX_CELLS + 1))
#define NA_CELL_PID (NA_CELL_FILL + NA_I32(CD_NOALLOC_MAX_CELLS))
#define NA_PCNT (NA_CELL_PID + NA_I32(CD_NOALLOC_MAX_N))
#define NA_POFF (NA_PCNT + NA_I32(CD_NOALLOC_MAX_N + 1))
#define NA_SCAN (NA_POFF + NA_I32(CD_NOALLOC_MAX_N + 1))
#define NA_MN (NA_SCAN + NA_I32(CD_NOALLOC_MAX_CELLS / 1024 + 64))
#define NA_MT (NA_MN + NA_ALIGN(sizeof(double) * CD_NOALLOC_MAX_CONTACTS))
#define NA_PK (NA_MT + NA_ALIGN(sizeof(double) * CD_NOALLOC_MAX_CONTACTS))
#define NA_CAND (NA_PK + NA_ALIGN(sizeof(double) * 4 * CD_NOALLOC_MAX_CONTACTS))
#define NA_TOT (NA_CAND + NA_I32((size_t)CD_NOALLOC_MAX_N * CD_CAND))
#define NA_PF (NA_TOT + NA_I32(4 * CD_PREP_MAX_BLOCKS))
#define NA_BYTES (NA_PF + NA_ALIGN(sizeof(float4) * CD_NOALLOC_MAX_N))

static __device__ __align__(256) unsigned char cd_noalloc_scratch[NA_BYTES];

// Of each device: the scratch array, and the launch plans (2D and 3D, by the
// size class of cd_prepare_plan).
static std::mutex na_mutex;
static void* na_addr[CD_NOALLOC_MAX_DEVICES];
static CdPrepPlan na_plan[CD_NOALLOC_MAX_DEVICES][2][2];

// Clears the control block, takes the largest radius (as ordered bits of a
// positive double; a flag if one is not positive and finite) and lays out the
// cell grid, by the operations of cd_create_system.  One block: n is small, and
// an atomic a particle on one address took 8 us of 5,000 particles' 112.  The
// grid used to be the host's, which had to wait for the radius first.
__global__ void __launch_bounds__(1024) k_noalloc_begin(CdCtrl* ctrl, CdGridSpec* grid, CdGeom g, double w0, double w1,
                                                        double w2, double w3, double w4, double w5,
                                                        const double* __restrict__ radius)
{
    __shared__ unsigned long long s_top[32];
    __shared__ int s_bad;
    __shared__ int s_m[3];
    if (threadIdx.x == 0) s_bad = 0;
    __syncthreads();
    unsigned long long top = 0ULL;
    bool bad = false;
    for (int i = threadIdx.x; i < g.n; i += blockDim.x) {
        const double r = radius[i];
        if (!(r > 0.0) || !isfinite(r)) bad = true;
        else top = max(top, (unsigned long long)__double_as_longlong(r));
    }
    if (bad) s_bad = 1;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
    if ((threadIdx.x & 31) == 0) s_top[threadIdx.x >> 5] = top;
    __syncthreads();
    if (threadIdx.x < 32) {
        top = s_top[threadIdx.x];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
        const double ell = __dmul_rn(__dadd_rn(__dmul_rn(2.0, __longlong_as_double((long long)top)), g.delta), 1.0 + 1e-9);
        const int k = threadIdx.x;
        if (k < 3) {
            double m = 1.0;
            if (k < g.dim) {
                m = floor(__ddiv_rn(g.L[k], ell));
                if (!(m >= 1.0)) m = 1.0;
                if (m > (double)CD_NOALLOC_MAX_CELLS) m = (double)CD_NOALLOC_MAX_CELLS;
                grid->cs[k] = __ddiv_rn(g.L[k], m);
                grid->inv_cs[k] = __ddiv_rn(1.0, grid->cs[k]);
            } else {
                grid->cs[k] = 1.0;
                grid->inv_cs[k] = 1.0;
            }
            grid->ncell[k] = s_m[k] = (int)m;
        }
        __syncwarp();
    }
    if (threadIdx.x == 0) {
        int status = s_bad ? CDG_RADIUS : CDG_OK;
        long long total = 1;
        for (int k = 0; k < 3; ++k) {
            if (g.periodic[k] && s_m[k] < 3 && status == CDG_OK) status = CDG_PERIODIC;
            total *= s_m[k];
        }
        if (total > CD_NOALLOC_MAX_CELLS && status == CDG_OK) status = CDG_CELLS;
        grid->total = total > CD_NOALLOC_MAX_CELLS ? CD_NOALLOC_MAX_CELLS : (int)total;
        grid->status = status;
        CdCtrl c;
        memset(&c, 0, sizeof c);
        c.wall_pos[0] = w0; c.wall_pos[1] = w1; c.wall_pos[2] = w2;
        c.wall_pos[3] = w3; c.wall_pos[4] = w4; c.wall_pos[5] = w5;
        *ctrl = c;
    }
}

// Message of a failure, read back with cd_last_error(NULL).
void cd_set_global_error(const char* msg);

static cd_status na_error(cd_status st, const char* msg)
{
    cd_set_global_error(msg);
    return st;
}

static cd_status na_cuda(cudaError_t e, const char* where)
{
    char buf[256];
    snprintf(buf, sizeof buf, "%s: %s", where, cudaGetErrorString(e));
    cd_set_global_error(buf);
    return CD_ERR_CUDA;
}

// What the call answers for what the device left behind (of the grid: CDG_*; of
// the control block: CDE_*, overflow, the count).  Not in the public header:
// apart from the call because the kernel's barriers have a bound, and what
// follows when one runs out is checked without making one run out.  The count
// is written where it is one.
extern "C" cd_status cd_noalloc_outcome(int grid, int error, int overflow, int nc_needed, int64_t* n_contacts)
{
    if (grid == CDG_RADIUS) return na_error(CD_ERR_INVALID_ARG, "radius must be positive and finite");
    if (grid == CDG_PERIODIC)
        return na_error(CD_ERR_INVALID_ARG, "a periodic axis needs at least 3 cells (box >= 3 l)");
    if (grid == CDG_CELLS)
        return na_error(CD_ERR_INVALID_ARG, "the box needs more than 65536 cells for the no-allocation entry point");
    if (error == CDE_TIMEOUT) return na_error(CD_ERR_TIMEOUT, "a bounded device-side wait ran out");
    *n_contacts = nc_needed;
    if (error == CDE_PER_PARTICLE) return na_error(CD_ERR_CAPACITY, "a particle has more than 64 contact candidates");
    if (error != CDE_NONE) return na_error(CD_ERR_STATE, "the detection failed on the device");
    if (overflow) return na_error(CD_ERR_CAPACITY, "more contacts than max_contacts; *n_contacts holds the number needed");
    return CD_OK;
}

extern "C" cd_status cd_detect_contacts_noalloc(const cd_params* params, int64_t n, const double* pos,
                                                const double* radius, const double* inv_mass,
                                                const double* inv_inertia, int64_t max_contacts, int32_t* pairs,
                                                double* normal, double* gap, int64_t* n_contacts, void* cuda_stream)
{
    cd_set_global_error("");
    if (!params || !pos || !radius || !inv_mass || !inv_inertia || !n_contacts)
        return na_error(CD_ERR_INVALID_ARG, "a required argument is NULL");
    const cd_params& p = *params;
    if (p.dim != 2 && p.dim != 3) return na_error(CD_ERR_INVALID_ARG, "dim must be 2 or 3");
    if (n <= 0 || n > CD_NOALLOC_MAX_N)
        return na_error(CD_ERR_INVALID_ARG, "particle count must be in [1, 16384] for the no-allocation entry point");
    if (max_contacts < 0 || max_contacts > CD_NOALLOC_MAX_CONTACTS)
        return na_error(CD_ERR_INVALID_ARG, "max_contacts must be in [0, 65536] for the no-allocation entry point");
    if (max_contacts > 0 && (!pairs || !normal || !gap))
        return na_error(CD_ERR_INVALID_ARG, "pairs, normal and gap are required when max_contacts > 0");
    if (!(p.dt > 0.0) || !(p.delta >= 0.0)) return na_error(CD_ERR_INVALID_ARG, "dt must be > 0 and delta >= 0");
    for (int k = 0; k < p.dim; ++k)
        if (!(p.box_hi[k] > p.box_lo[k])) return na_error(CD_ERR_INVALID_ARG, "box_hi must exceed box_lo");
    for (int k = 0; k < 6; ++k)
        if (((p.wall_mask >> k) & 1) && ((k >> 1) >= p.dim || p.periodic[k >> 1]))
            return na_error(CD_ERR_INVALID_ARG, "wall on a missing or periodic axis");
    cudaStream_t s = (cudaStream_t)cuda_stream;

    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return na_cuda(e, "cudaGetDevice");
    if (dev < 0 || dev >= CD_NOALLOC_MAX_DEVICES) return na_error(CD_ERR_INVALID_ARG, "device index out of range");
    unsigned char* base = nullptr;
    CdPrepPlan plan;
    {
        std::lock_guard<std::mutex> lock(na_mutex);
        if (!na_addr[dev]) {
            void* ptr = nullptr;
            e = cudaGetSymbolAddress(&ptr, cd_noalloc_scratch);
            if (e != cudaSuccess) return na_cuda(e, "cudaGetSymbolAddress");
            na_addr[dev] = ptr;
        }
        base = (unsigned char*)na_addr[dev];
        CdPrepPlan& known = na_plan[dev][p.dim - 2][n <= cd_prepare_cluster_n((int)p.dim) ? 1 : 0];
        if (!known.blocks) known = cd_prepare_plan((int)p.dim, CD_FP64, 1, n, CD_NOALLOC_MAX_CELLS, dev);
        plan = known;
    }
    if (!plan.blocks) return na_error(CD_ERR_CUDA, "the detection kernel does not fit on this device");

    CdCtrl* ctrl = (CdCtrl*)(base + NA_CTRL);
    CdGridSpec* grid = (CdGridSpec*)(base + NA_GRID);
    CdGeom g;
    memset(&g, 0, sizeof g);
    g.dim = (int)p.dim;
    g.n = (int)n;
    g.cap = (int)max_contacts;
    g.wall_mask = (int)p.wall_mask;
    g.delta = p.delta;
    g.dt = p.dt;
    g.mu = p.mu;
    g.rotations = (int)p.rotations;
    g.seed = p.seed;
    g.npk = 1;
    for (int k = 0; k < 3; ++k) {
        g.periodic[k] = (k < p.dim) ? (int)p.periodic[k] : 0;
        g.lo[k] = (k < p.dim) ? p.box_lo[k] : 0.0;
        g.hi[k] = (k < p.dim) ? p.box_hi[k] : 1.0;
        g.L[k] = (k < p.dim) ? p.box_hi[k] - p.box_lo[k] : 1.0;
    }
    k_noalloc_begin<<<1, 1024, 0, s>>>(ctrl, grid, g, p.wall_pos[0], p.wall_pos[1], p.wall_pos[2], p.wall_pos[3],
                                       p.wall_pos[4], p.wall_pos[5], radius);

    CdWork w;
    memset(&w, 0, sizeof w);
    w.ctrl = ctrl;
    w.cell_of = (int*)(base + NA_CELL_OF);
    w.cell_cnt = (int*)(base + NA_CELL_CNT);
    w.cell_start = (int*)(base + NA_CELL_START);
    w.cell_fill = (int*)(base + NA_CELL_FILL);
    w.cell_pid = (int*)(base + NA_CELL_PID);
    w.pcnt = (int*)(base + NA_PCNT);
    w.poff = (int*)(base + NA_POFF);
    w.cand = (int*)(base + NA_CAND);
    w.pf = (float4*)(base + NA_PF);
    w.scan_tmp = (int*)(base + NA_SCAN);
    w.mn = (double*)(base + NA_MN);
    w.mt = (double*)(base + NA_MT);
    w.Pk_nx = (double*)(base + NA_PK);
    w.Pk = w.Pk_nx;                 // the commit copy runs in place
    w.pairs_nx = (int2*)pairs;      // caller outputs
    w.pairs = (int2*)pairs;
    w.nrm = normal;
    w.gap = gap;
    w.pk_wall_pos = ctrl->wall_pos;   // device address inside the scratch
    const int pw = (p.dim == 2) ? 2 : 4;
    int nl = 0;
    w.prep_tot = (int*)(base + NA_TOT);
    CdPrepIO io = {};
    io.pos = pos; io.radius = radius; io.inv_m = inv_mass; io.inv_I = inv_inertia;
    io.pw = pw;
    io.grid = grid;
    if ((e = cd_launch_prepare(g, w, io, plan.blocks, plan.cluster, CD_FP64, s, &nl)) != cudaSuccess)
        return na_cuda(e, "detection launch");
    alignas(16) unsigned char back[NA_GRID + sizeof(CdGridSpec)];
    if ((e = cudaMemcpyAsync(back, base, sizeof back, cudaMemcpyDeviceToHost, s)) != cudaSuccess)
        return na_cuda(e, "reading the contact count");
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return na_cuda(e, "cudaStreamSynchronize");
    CdCtrl h;
    CdGridSpec hg;
    memcpy(&h, back + NA_CTRL, sizeof h);
    memcpy(&hg, back + NA_GRID, sizeof hg);
    return cd_noalloc_outcome(hg.status, h.error, h.overflow, h.nc_needed, n_contacts);
}
