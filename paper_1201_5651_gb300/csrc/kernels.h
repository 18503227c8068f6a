// Kernel launch interfaces used by the host driver.
#pragma once
#include <cuda_runtime.h>
#include <limits.h>
#include "oots_internal.h"

#ifdef __CUDACC__
#define OOTS_HOSTDEV __host__ __device__
#else
#define OOTS_HOSTDEV
#endif

namespace oots {

template <typename Real> struct DevTable;
struct ff;
template <typename Real> struct ColT;

// The tile shapes of oots_set_tile_shape.  The marches below have blocks of
// their own, so the shapes only keep their meaning at the interface: dims, and
// the one that FP64 refuses (its tile once needed more shared memory than a
// block has).
enum { NUM_SHAPES = 9, SHAPE_16_CUBED = 2 };
static const int SHAPE_DIMS[NUM_SHAPES][3] = {{16, 8, 8}, {16, 8, 4}, {16, 16, 16}, {32, 8, 4}, {8, 8, 8},
                                              {16, 16, 8}, {8, 8, 4}, {8, 8, 8}, {16, 8, 8}};

// The column march (march.cuh).  A published cell is one 16-byte record: its
// outgoing column (float-float in the mixed path) and weight factor.
template <typename Real> struct MCell;
template <> struct alignas(16) MCell<float> { float hi, lo, w, pad; };
template <> struct alignas(16) MCell<double> { double n, w; };

template <typename Real> struct MarchParams {
    const GridDev<Real> *grids;
    const March *marches;
    const MarchItem *items;            // in the order they are handed out
    int nitems;
    int which;                         // 0: trace x into N1; 1: trace xh into N2
    unsigned *ticket, *done;           // zero before each launch (the launch leaves them so)
    unsigned *epoch;                   // launches finished so far (persistent; starts at 0)
    const DevTable<Real> *tabs;        // A1
    MCell<Real> *halo;
    unsigned long long *progress;      // per item: chunks of layers published, tagged with the launch's epoch
    int *err;                          // sticky device error
    long long spin_limit;              // bounded wait on upstream items
    long long ready_limit;             // and on the CTA's own handing warp (march_ready_limit)
    long long skip_publish;            // item that never publishes (fault-injection test), -1: none
    int ngrid;                         // grids in `grids` (> 0: the launch returns at once when every
                                       // grid has reached its end time; 0: no such check)
    int narr;                          // input arrays of a cell: 1 (x or n x packed), 2 when some grid brings n and x
};

// Blocks of the march: 32 x ROWS cells, NW warps of RPT rows (the measurements are in march.cuh).
template <typename Real> struct MarchShape { enum { NW = 7, RPT = sizeof(Real) == 4 ? 3 : 1, ROWS = NW * RPT }; };
constexpr int kMarchChunk = 8;       // layers of a trace between two progress publications
// Limits of the waits inside a CTA of the march.  The handing warp waits for other CTAs (spin_limit polls)
// and gives up alone: what its computing warps wait for comes after that at the latest, so their limit, in
// tests of at least ten nanoseconds, lies a thousand times its polls of about half a microsecond above it.
// A chunk of layers takes milliseconds at most (A1: of front cells in FP64), the limit on it is a second or more.
OOTS_HOSTDEV inline long long march_ready_limit(long long spin_limit)
{
    return spin_limit < ((LLONG_MAX - (1 << 24)) >> 10) ? (spin_limit << 10) + (1 << 24) : LLONG_MAX;
}
constexpr int kMarchDoneLimit = 1 << 24;
// sets the kernel up on the current device; CTAs per SM with narr input arrays
template <typename Real> cudaError_t march_occupancy(int narr, int *per_sm);
template <typename Real>
cudaError_t launch_march(const MarchParams<Real> &P, int nblocks, cudaStream_t s);
// A1 (march_a1.cuh): blocks of 32 x kMarchA1Warps cells; reads the state from GridDev::xh, writes xout
constexpr int kMarchA1Warps = 7;
template <typename Real> cudaError_t march_a1_occupancy(int *per_sm);
template <typename Real>
cudaError_t launch_march_a1(const MarchParams<Real> &P, int nblocks, cudaStream_t s);
// n x of the traced state (which = 0: x, 1: xh) into each grid's padded rows (GridDev::nxp);
// max_elems = the largest grid's padded cells
template <typename Real>
cudaError_t launch_pack_nx(const GridDev<Real> *grids, int ngrid, int which, long long max_elems, int nsm,
                           cudaStream_t s);

// The pyramid of `axis` in octant o (bit a set: the side below the vertex along
// axis a) of a source at vertex v; false when the octant is empty.  pitch: row
// length of the input (nx unless packed).
OOTS_HOSTDEV inline bool make_march(March &M, int nx, int ny, int nz, const int v[3], int o, int axis, int pitch,
                                    bool packed)
{
    const int n3[3] = {nx, ny, nz};
    int sg[3], ext[3];
    long long c0[3];
    for (int a = 0; a < 3; a++) {
        sg[a] = (o >> a) & 1 ? -1 : 1;
        ext[a] = sg[a] > 0 ? n3[a] - v[a] : v[a];
        if (ext[a] <= 0) return false;
        c0[a] = sg[a] > 0 ? v[a] : v[a] - 1;
    }
    const int au = axis == 0 ? 1 : 0, aw = axis == 2 ? 1 : 2;
    const long long is[3] = {1, pitch, (long long)pitch * ny}, os[3] = {1, nx, (long long)nx * ny};
    M.grid = M.src = 0;
    M.axis = axis;
    M.sg = sg[0];
    M.len = ext[axis];
    M.eu = ext[au];
    M.ew = ext[aw];
    M.off = axis == 0 ? (sg[0] > 0 ? v[0] % 8 : (8 - v[0] % 8) % 8) : 0;
    M.packed = packed;
    M.pad[0] = M.pad[1] = M.pad[2] = 0;
    M.ibase = c0[0] + c0[1] * is[1] + c0[2] * is[2];
    M.obase = c0[0] + c0[1] * os[1] + c0[2] * os[2];
    M.isl = sg[axis] * is[axis]; M.isu = sg[au] * is[au]; M.isw = sg[aw] * is[aw];
    M.osl = sg[axis] * os[axis]; M.osu = sg[au] * os[au]; M.osw = sg[aw] * os[aw];
    return true;
}
// blocks of a pyramid along u and w
OOTS_HOSTDEV inline int march_nt1(const March &M) { return ((M.eu < M.len ? M.eu : M.len) + 31) / 32; }
OOTS_HOSTDEV inline int march_nt2(const March &M, int rows) { return ((M.ew < M.len ? M.ew : M.len) + rows - 1) / rows; }
// Layers an item publishes: [first, len) of its pyramid, first = its l0.  A chunk is staged whole, also
// where its first layers lie before the neighbour's and its last ones beyond the pyramid: those are no
// cells of the halo.
OOTS_HOSTDEV inline bool march_published(int l, int first, int len) { return l >= first && l < len; }
// block (T1, T2) without its neighbours' item numbers and halo; returns the cells it publishes
OOTS_HOSTDEV inline long long make_march_item(MarchItem &I, const March &M, int march, int T1, int T2, int rows)
{
    I.march = march;
    I.T1 = (unsigned short)T1;
    I.T2 = (unsigned short)T2;
    I.l0 = 32 * T1 > rows * T2 ? 32 * T1 : rows * T2;
    I.right = T1 + 1 < march_nt1(M);
    I.above = T2 + 1 < march_nt2(M, rows);
    I.pad = 0;
    I.pad2 = 0;
    I.up0 = I.up1 = I.up2 = -1;
    I.halo = 0;
    return I.right || I.above ? (long long)(M.len - I.l0) * (rows + 32) : 0;
}

// Plane-parallel sources: which = 0 traces x into N1, 1 traces xh into N2;
// implicit = 1 runs the A1 row integration instead (single source).  The jobs
// along x come first (nrow0 of them, threads0 threads); nthreads is the sum
// of plane_job_threads over all jobs, whose `first` fields are the running
// sums.  rows0: the first job's rows (A1's only source).
long long plane_job_threads(int code, long long rows);
template <typename Real>
cudaError_t launch_plane(const GridDev<Real> *grids, const PlaneJob *jobs, int njobs, int nrow0, long long nthreads,
                         long long threads0, long long rows0, const DevTable<Real> *tabs, int which, int implicit, cudaStream_t s);

// Per-cell passes.  HALF and FULL run as a closed-form pass over all cells
// followed by the general pass (op | OP_GENERAL) over the queued cells.
enum { OP_RATEDT = 0, OP_HALF = 1, OP_FULL1 = 2, OP_FULL2 = 3, OP_RATEDT_VERIFY = 4, OP_GENERAL = 16 };
// qrec: per queue slot the closed-form pass's rates and f(x0) of single-source
// cells (queue_record_bytes each), so the general pass starts at the root
// search (unused, may be null, when nsmax > 1).  rcache: 3 x total values per
// cell that the dt pass writes and the half step (A3) or full step (A2) of
// the same substep reads when use_cache is set: the transmitted fraction,
// F(x0) and F'(x0) of single-source grids; F(x0), F'(x0) and the sum of the
// sources' rate bounds when nsmax > 1 (the full step then recomputes).
// cell_bs: threads per block of the closed-form passes, 128 or 256 (the general passes use 256).
template <typename Real>
cudaError_t launch_cell(const GridDev<Real> *grids, int ngrid, const long long *offsets, long long total,
                        const DevTable<Real> *tabs, int op, int nsmax, unsigned *queue, unsigned *qcount,
                        Real *qrec, Real *rcache, int use_cache, int gen_blocks, int cell_bs, cudaStream_t s);
template <typename Real> size_t queue_record_bytes();
template <typename Real> int cell_general_occupancy(int nsmax);
// stage 0 also clears the queue lengths and the general passes' head counters
template <typename Real>
cudaError_t launch_finalize(const GridDev<Real> *grids, int ngrid, int stage, unsigned *qcount,
                            const DevTable<Real> *tabs, cudaStream_t s);

} // namespace oots
