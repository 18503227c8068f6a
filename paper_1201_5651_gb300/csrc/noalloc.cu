// oots_trace_noalloc: the column-density trace for callers that cannot
// allocate device memory.  It runs the same trace kernel as the
// context API, but every piece of scratch it needs (the work list, the
// halos between blocks and the small descriptors) lives in one file-scope static device array, so the call makes no cudaMalloc, no
// cudaFree and no heap allocation on the host.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>

#include <cuda_runtime.h>

#include "../../include/oots.h"
#include "common.cuh"
#include "kernels.h"

using namespace oots;

// error text for oots_last_error (defined with the rest of the C ABI)
void oots_set_error_text(const char *msg);

namespace {

// 64 MiB, resident on every device that loads the library until the process exits.
constexpr size_t kScratchBytes = (size_t)64 << 20;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

// The size limit is stated in tiles of 16 x 8 x 8 cells.
constexpr int kTX = 16, kTY = 8, kTZ = 8;
constexpr int kMaxDiag = 4096;                  // tile diagonals within the limit
constexpr int kMaxMarch = 24;                   // pyramids of one source
constexpr int kMaxItems = 4096;                 // blocks of all pyramids (a grid within the limit has under a thousand)
constexpr int kMaxItemDiag = 2048;              // block diagonals T1 + T2 of a pyramid (sides up to 8192)

// header layout (byte offsets inside the scratch)
constexpr size_t kOffTicket = 0;                // ticket, then the count of finished CTAs
constexpr size_t kOffEpoch = 64;                // marches so far: never cleared (progress words carry it)
constexpr size_t kOffErr = 128;
constexpr size_t kOffState = 256;               // DevState (done = 0 after the clear)
constexpr size_t kOffCount = 1024;              // kMaxItemDiag unsigned: items per diagonal, then cursors
constexpr size_t kOffMarch = kOffCount + 2 * kMaxItemDiag * sizeof(unsigned) + 256;
constexpr size_t kOffGrid = kOffMarch + kMaxMarch * sizeof(March) + 256;

struct DevSetup {
    bool ready = false;
    unsigned char *scratch = nullptr;
    int nblocks[2][2] = {};   // per precision and number of input arrays
};
static DevSetup g_setup[64];
static std::mutex g_setup_mutex;   // first-call set-up of a device, from any host thread

// Byte offset of the per-item arrays, and the most tiles a grid may have: the
// limit this entry point has always stated.  The march needs far less (its
// published cells are a twentieth of the tiles' faces); the call checks it.
template <typename Real> size_t items_offset()
{
    return (kOffGrid + sizeof(GridDev<Real>) + 255) / 256 * 256;
}
template <typename Real> long long max_tiles();
template <> long long max_tiles<float>() { return 7264; }
template <> long long max_tiles<double>() { return 5450; }

struct MarchSet {
    March m[kMaxMarch];
    int n;
};

// One block lists the items of the (at most 24) pyramids by block diagonal:
// count per diagonal, exclusive scan, then place (order inside a diagonal is
// free), then each item's neighbours.
template <typename Real>
__global__ void build_worklist(const __grid_constant__ MarchSet S, const __grid_constant__ GridDev<Real> G0,
                               unsigned char *sc, int rows, MarchItem *items, int *at, int maxdiag)
{
    unsigned *count = (unsigned *)(sc + kOffCount), *cursor = count + kMaxItemDiag;
    March *marches = (March *)(sc + kOffMarch);
    __shared__ unsigned s_halo;                 // published cells so far (below 2^32: 64 MiB of 16-byte cells)
    if (threadIdx.x == 0) {
        s_halo = 0u;
        *(GridDev<Real> *)(sc + kOffGrid) = G0;
        *(int *)(sc + kOffErr) = 0;
        // (a launch leaves these zero, but one cut across by another call may not have)
        ((unsigned *)(sc + kOffTicket))[0] = 0u;
        ((unsigned *)(sc + kOffTicket))[1] = 0u;
        DevState *st = (DevState *)(sc + kOffState);
        st->done = 0;
    }
    for (int j = threadIdx.x; j < S.n; j += blockDim.x) marches[j] = S.m[j];
    for (int d = threadIdx.x; d < maxdiag; d += blockDim.x) { count[d] = 0u; cursor[d] = 0u; }
    __syncthreads();
    for (int j = 0; j < S.n; j++) {
        const int n1 = march_nt1(S.m[j]), n = n1 * march_nt2(S.m[j], rows);
        for (int t = threadIdx.x; t < n; t += blockDim.x) atomicAdd(&count[t % n1 + t / n1], 1u);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned acc = 0;
        for (int d = 0; d < maxdiag; d++) { const unsigned c = count[d]; cursor[d] = acc; acc += c; }
    }
    __syncthreads();
    int first = 0;
    for (int j = 0; j < S.n; j++) {
        const int n1 = march_nt1(S.m[j]), n = n1 * march_nt2(S.m[j], rows);
        for (int t = threadIdx.x; t < n; t += blockDim.x) {
            MarchItem I;
            const unsigned pub = (unsigned)make_march_item(I, S.m[j], j, t % n1, t / n1, rows);
            const unsigned pos = atomicAdd(&cursor[t % n1 + t / n1], 1u);
            I.halo = atomicAdd(&s_halo, pub);
            items[pos] = I;
            at[first + t] = (int)pos;
        }
        first += n;
    }
    __syncthreads();
    first = 0;
    for (int j = 0; j < S.n; j++) {
        const int n1 = march_nt1(S.m[j]), n = n1 * march_nt2(S.m[j], rows);
        for (int t = threadIdx.x; t < n; t += blockDim.x) {
            MarchItem &I = items[at[first + t]];
            const int T1 = t % n1, T2 = t / n1;
            if (T1 > 0) I.up0 = at[first + t - 1];
            if (T2 > 0) I.up1 = at[first + t - n1];
            if (T1 > 0 && T2 > 0) I.up2 = at[first + t - n1 - 1];
        }
        first += n;
    }
}

template <typename Real>
int trace_noalloc(DevSetup &S, int nx, int ny, int nz, double dx, const void *n_dev, double n_uniform,
                  const void *x_dev, const int vtx[3], double sigma0, double tau0, void *Nin_dev, cudaStream_t st)
{
    const int n3[3] = {nx, ny, nz};
    const int T3[3] = {kTX, kTY, kTZ};
    long long tiles = 0;
    int maxd = 0;
    for (int o = 0; o < 8; o++) {
        int nt[3];
        bool empty = false;
        for (int a = 0; a < 3; a++) {
            const int ext = (o >> a) & 1 ? vtx[a] : n3[a] - vtx[a];
            if (ext <= 0) empty = true;
            const int r = vtx[a] % T3[a];
            const int off = (o >> a) & 1 ? (T3[a] - r) % T3[a] : r;
            nt[a] = (ext + off + T3[a] - 1) / T3[a];
        }
        if (empty) continue;
        tiles += (long long)nt[0] * nt[1] * nt[2];
        maxd = std::max(maxd, nt[0] + nt[1] + nt[2] - 2);
    }
    const long long maxt = max_tiles<Real>();
    if (tiles > maxt || maxd + 1 > kMaxDiag)
        return -1000 - (int)std::min<long long>(tiles, 1 << 30);   // reported by the caller

    GridDev<Real> G;
    memset(&G, 0, sizeof(G));
    unsigned char *sc = S.scratch;
    G.nx = nx; G.ny = ny; G.nz = nz;
    G.ncell = (long long)nx * ny * nz;
    G.cell_lo = 0;
    G.cell_hi = G.ncell;
    G.dx = Real(dx);
    G.sigma0 = Real(sigma0);
    G.tau0 = Real(tau0);
    G.n = (const Real *)n_dev;
    G.n_uniform = Real(n_uniform);
    G.x = (const Real *)x_dev;
    G.xh = (const Real *)x_dev;
    G.N1 = (Real *)Nin_dev;
    G.nsrc = 1;
    for (int a = 0; a < 3; a++) G.vtx[0][a] = vtx[a];
    G.tab[0] = -1;
    G.pitch = nx;
    G.st = (DevState *)(sc + kOffState);

    MarchSet set;
    set.n = 0;
    for (int o = 0; o < 8; o++)
        for (int a = 0; a < 3; a++)
            if (make_march(set.m[set.n], nx, ny, nz, vtx, o, a, nx, false)) set.n++;
    const int narr = n_dev ? 2 : 1;
    const int rows = MarchShape<Real>::ROWS;
    long long nitems = 0, cells = 0;
    int itemdiag = 0;
    for (int j = 0; j < set.n; j++) {
        const int n1 = march_nt1(set.m[j]), n2 = march_nt2(set.m[j], rows);
        nitems += (long long)n1 * n2;
        itemdiag = std::max(itemdiag, n1 + n2 - 1);
        for (int t = 0; t < n1 * n2; t++) {
            MarchItem I;
            cells += make_march_item(I, set.m[j], j, t % n1, t / n1, rows);
        }
    }
    // the per-item arrays after the fixed part: progress words first (they must
    // keep the tags of earlier launches, so their place does not move)
    size_t off = items_offset<double>();
    unsigned long long *progress = (unsigned long long *)(sc + off);
    off += kMaxItems * sizeof(unsigned long long);
    MarchItem *items = (MarchItem *)(sc + off);
    off += kMaxItems * sizeof(MarchItem);
    int *at = (int *)(sc + off);
    off += kMaxItems * sizeof(int);
    MCell<Real> *halo = (MCell<Real> *)(sc + off);
    if (nitems > kMaxItems || itemdiag > kMaxItemDiag || off + (size_t)cells * sizeof(MCell<Real>) > kScratchBytes)
        return -1000 - (int)std::min<long long>(tiles, 1 << 30);
    if (nitems == 0) return 0;
    build_worklist<Real><<<1, 1024, 0, st>>>(set, G, sc, rows, items, at, itemdiag);
    if (cudaGetLastError() != cudaSuccess) return -1;

    MarchParams<Real> P;
    P.grids = (const GridDev<Real> *)(sc + kOffGrid);
    P.marches = (const March *)(sc + kOffMarch);
    P.items = items;
    P.nitems = (int)nitems;
    P.which = 0;
    P.ticket = (unsigned *)(sc + kOffTicket);
    P.done = (unsigned *)(sc + kOffTicket) + 1;
    P.epoch = (unsigned *)(sc + kOffEpoch);
    P.tabs = nullptr;
    P.halo = halo;
    P.progress = progress;
    P.err = (int *)(sc + kOffErr);
    P.spin_limit = 1ll << 22;
    P.ready_limit = march_ready_limit(P.spin_limit);
    P.skip_publish = -1;
    P.ngrid = 0;
    P.narr = narr;
    const int prec = sizeof(Real) == 8 ? 0 : 1;
    if (launch_march<Real>(P, S.nblocks[prec][narr - 1], st) != cudaSuccess) return -1;
    return 0;
}

} // namespace

extern "C" int oots_trace_noalloc(int device, int precision, int nx, int ny, int nz, double dx_cm,
                                  const void *n_dev, double uniform_n, const void *x_dev, const double pos_cells[3],
                                  double sigma0, double tau0, void *Nin_dev, void *stream, int *status_detail)
{
    if (status_detail) *status_detail = 0;
    if (precision != OOTS_FP64 && precision != OOTS_MIXED) return OOTS_E_INVAL;
    if (nx <= 0 || ny <= 0 || nz <= 0 || nx > 8192 || ny > 8192 || nz > 8192) return OOTS_E_INVAL;
    if (!(dx_cm > 0) || !std::isfinite(dx_cm) || !(sigma0 > 0) || !(tau0 > 0)) return OOTS_E_INVAL;
    if (!x_dev || !Nin_dev || !pos_cells) return OOTS_E_INVAL;
    if (!n_dev && !(uniform_n > 0)) return OOTS_E_INVAL;
    if (device < 0 || device >= 64) return OOTS_E_INVAL;
    int vtx[3];
    const int n3[3] = {nx, ny, nz};
    for (int a = 0; a < 3; a++) {
        if (!std::isfinite(pos_cells[a])) return OOTS_E_INVAL;
        double v = std::floor(pos_cells[a] + 0.5);
        vtx[a] = (int)std::min<double>(std::max<double>(v, 0.0), n3[a]);
    }
    int prev = 0;
    if (cudaGetDevice(&prev) != cudaSuccess) return OOTS_E_CUDA;
    if (cudaSetDevice(device) != cudaSuccess) return OOTS_E_CUDA;
    DevSetup &S = g_setup[device];
    int rc = OOTS_OK;
    std::unique_lock<std::mutex> setup_lock(g_setup_mutex);
    if (!S.ready) {
        // once per device, with the device current: the device address of the
        // static scratch (its host-side name is only a stand-in) and the
        // persistent grid sizes
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) rc = OOTS_E_CUDA;
        if (rc == OOTS_OK) {
            int nsm = 0;
            cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, device);
            S.scratch = (unsigned char *)p;
            for (int a = 0; a < 2 && rc == OOTS_OK; a++) {
                int o64 = 0, o32 = 0;
                if (march_occupancy<double>(a + 1, &o64) != cudaSuccess || march_occupancy<float>(a + 1, &o32) != cudaSuccess)
                    rc = OOTS_E_CUDA;
                S.nblocks[0][a] = o64 * nsm;
                S.nblocks[1][a] = o32 * nsm;
            }
            S.ready = rc == OOTS_OK;
        }
    }
    setup_lock.unlock();
    cudaStream_t st = (cudaStream_t)stream;
    if (rc == OOTS_OK) {
        int r = precision == OOTS_FP64
                    ? trace_noalloc<double>(S, nx, ny, nz, dx_cm, n_dev, uniform_n, x_dev, vtx, sigma0, tau0, Nin_dev, st)
                    : trace_noalloc<float>(S, nx, ny, nz, dx_cm, n_dev, uniform_n, x_dev, vtx, sigma0, tau0, Nin_dev, st);
        if (r <= -1000) {
            if (status_detail) *status_detail = -1000 - r;   // tiles the problem needs
            char msg[256];
            snprintf(msg, sizeof(msg),
                     "oots_trace_noalloc: the grid needs %d tiles of 16x8x8 cells; the %zu MiB static scratch holds "
                     "at most %lld (%s)", -1000 - r, kScratchBytes >> 20,
                     precision == OOTS_FP64 ? max_tiles<double>() : max_tiles<float>(),
                     precision == OOTS_FP64 ? "FP64" : "mixed");
            oots_set_error_text(msg);
            rc = OOTS_E_INVAL;
        } else if (r != 0) {
            rc = OOTS_E_CUDA;
        } else {
            int err = 0;
            if (cudaMemcpyAsync(&err, S.scratch + kOffErr, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
                cudaStreamSynchronize(st) != cudaSuccess)
                rc = OOTS_E_CUDA;
            else if (err == DEVERR_TIMEOUT)
                rc = OOTS_E_DEVICE_TIMEOUT;
        }
    }
    cudaSetDevice(prev);
    return rc;
}
