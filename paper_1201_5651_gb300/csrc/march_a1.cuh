// The implicit scheme's march (Mackey 2012, Sect. 2.1, A1): the column march
// (march.cuh: pyramids per dominant axis, blocks of 32 x 7 cells, one barrier
// per layer, halos handed over per chunk) with every cell integrated on the
// way, its entry column frozen, handing downstream N_in - ln<f>/sigma0 from its
// time-averaged attenuation <f> (Eq. 3).
//
// A layer lasts as long as its slowest cell.  Each lane settles its own cell
// when a closed form covers it (photon-free, slow, next to its root: all but
// those the front crosses).  A few others are taken by lane groups (a half
// warp each, FP64 a warp), the nodes of every quadrature panel spread over the
// lanes; more of them, where the front runs along a row, by one lane each.  x
// is read from a copy made before the launch:
// tied cells belong to several pyramids, all integrate them, one writes them.
//
// What bounds it: the chain of layers, each as long as its slowest warp (0.5 ms
// for a warp whose 32 cells the front crosses, 15 us for a single such cell).
// 88^3 cells, source in a corner (mixed): 44.5 -> 7.5 ms against tiles swept
// along i + j + k with every cell integrated by its own thread (262 planes in
// a row in place of 88 layers; with the series step of slow cells that sweep
// took 20.6 ms).  Chunks of eight layers: 21 ms (a block follows its neighbours
// one chunk behind), of two 7.9 ms; always a lane per cell 7.7 ms, always lane
// groups 11.8 ms.
#pragma once
#include "march.cuh"
#include "integrator.cuh"

namespace oots {

// layers between two progress publications: a block follows its neighbours one
// chunk behind, and a layer is long here
constexpr int kA1Chunk = 1;
// rounds of lane groups that are still shorter than one cell per lane
constexpr int kA1Groups = 2;

// Cells of a warp that the closed forms left, by lane groups.  R: this lane's
// result (its prelude's defaults on entry where `general` is set).
template <typename Real>
__device__ __forceinline__ void a1_general(bool general, const CellODE<Real> &C, Real x0, Real h, Real sigma0,
                                           Real F0, Real dF0, Real f0, IntResult<Real> &R)
{
    constexpr int W = GroupWidth<Real>::value, NG = 32 / W;
    const int lane = threadIdx.x & 31, grp = lane / W, base = grp * W;
    const unsigned gmask = W == 32 ? 0xffffffffu : (0xffffu << base);
    unsigned todo = __ballot_sync(0xffffffffu, general);
    if (__popc(todo) > kA1Groups * NG) {
        // many cells (the front crosses the row): every lane its own
        if (general) R = integrate_general<Real, 1>(C, x0, h, sigma0, R, F0, dF0, f0, SeqEval());
        __syncwarp();
        return;
    }
    while (todo) {
        // the next NG cells of the warp, one per group (a group without one repeats the last)
        int src[NG];
        unsigned t = todo;
#pragma unroll
        for (int k = 0; k < NG; k++) {
            src[k] = t ? __ffs(t) - 1 : src[k > 0 ? k - 1 : 0];
            t &= t - 1u;
        }
        const int s = src[NG - 1 < grp ? NG - 1 : grp];
        SrcRate<Real> r;
        CellODE<Real> D;
        const SrcRate<Real> &r0 = C.r[0];
        r.A = __shfl_sync(0xffffffffu, r0.A, s);
        r.b = __shfl_sync(0xffffffffu, r0.b, s);
        r.Nin = __shfl_sync(0xffffffffu, r0.Nin, s);
        r.p = __shfl_sync(0xffffffffu, r0.p, s);
        r.tab = __shfl_sync(0xffffffffu, r0.tab, s);
        D.ns = 1;
        D.c = __shfl_sync(0xffffffffu, C.c, s);
        D.b0 = __shfl_sync(0xffffffffu, C.b0, s);
        D.r = &r;
        D.tabs = C.tabs;
        IntResult<Real> Q;
        const Real gx0 = __shfl_sync(0xffffffffu, x0, s);
        const Real gF0 = __shfl_sync(0xffffffffu, F0, s), gdF0 = __shfl_sync(0xffffffffu, dF0, s);
        const Real gf0 = __shfl_sync(0xffffffffu, f0, s);
        Q.x = gx0; Q.IR = Real(0); Q.lnfav = -D.b0 * gx0;
        Q = integrate_general<Real, 1>(D, gx0, h, sigma0, Q, gF0, gdF0, gf0, GroupEval<W, true>{lane - base, base, gmask});
        __syncwarp();
#pragma unroll
        for (int k = 0; k < NG; k++) {
            const Real x = __shfl_sync(0xffffffffu, Q.x, k * W), ir = __shfl_sync(0xffffffffu, Q.IR, k * W);
            const Real ln = __shfl_sync(0xffffffffu, Q.lnfav, k * W);
            if (lane == src[k]) { R.x = x; R.IR = ir; R.lnfav = ln; }
            todo &= ~(1u << src[k]);
        }
    }
}

template <typename Real, int NW>
__device__ __forceinline__ void march_a1_item(const MarchParams<Real> &P, const MarchItem &it, const March &M,
                                              const GridDev<Real> &G, int c0, int c1, unsigned &phase,
                                              MarchShared<Real, NW, 1, kA1Chunk> &S)
{
    typedef MarchLayout<Real, NW, 1> L;
    typedef typename ColT<Real>::type Col;
    constexpr int B = L::B, H = kA1Chunk;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int u = it.T1 * 32 + lane, w = it.T2 * B + warp;
    const int l0 = it.l0, len = M.len, axis = M.axis, s = M.src, tab = G.tab[M.src];
    const Real sig = G.sigma0, tau0 = G.tau0, dx = G.dx, qfac = G.qfac[M.src], alpha = G.alpha, nu = G.n_uniform;
    const Real *nd = G.n;
    const Real *xs = G.xh;                               // the copy of x made before the launch
    Real *xout = G.xout, *Nout = G.N1 + (long long)s * G.ncell;
    const Real dt = Real(G.st->dt);
    const double cellV = G.st->cell_volume;
    const bool in = u < M.eu && w < M.ew;
    const long long sl = axis == 0 ? (long long)M.sg : M.osl, su = axis == 0 ? M.osu : (long long)M.sg;
    const int lf = c0 * H;
    long long g = M.obase + u * su + w * M.osw + lf * sl;
    MCell<Real> *phalo = P.halo + it.halo + (long long)(lf - l0) * L::STRIDE;
    const bool pub_r = it.right && lane == 31, pub_a = it.above && warp == NW - 1;
    Col N = ColT<Real>::zero();
    Real W = Real(1);
    double ions = 0.0, rec = 0.0;
    for (int c = c0; c <= c1; c++, phase++) {
        const int b = (int)(phase & 1u);
        march_await(P, S, phase);
        for (int q = 0; q < H; q++, g += sl, phalo += L::STRIDE) {
            const int l = c * H + q;
            if (l < l0 || l >= len) continue;
            const bool act = in && u <= l && w <= l;
            const Real n = act ? (nd ? __ldg(nd + g) : nu) : Real(1), x0 = act ? __ldg(xs + g) : Real(1);
            // entry column: the neighbours and weights of march_item
            const bool e1 = u >= l, e2 = w >= l;
            const Real ica = Real(1) / Real(2 * l + 1);
            const Real g1 = e1 ? Real(1) : Real(2 * u + 1) * ica, g2 = e2 ? Real(1) : Real(2 * w + 1) * ica;
            const Real p1 = Real(1) - g1, p2 = Real(1) - g2;
            const MCell<Real> bel = warp > 0 ? S.row[(l + 1) & 1][warp > 0 ? warp - 1 : 0][lane] : S.bot[b][q][lane + 1];
            MCell<Real> bel_l = mc_up(bel);
            mc_lane0(bel_l, warp > 0 ? &S.left[b][q][warp > 0 ? warp - 1 : 0] : &S.bot[b][q][0], lane);
            MCell<Real> lef = mc_up(mc_make(N, W));
            mc_lane0(lef, &S.left[b][q][warp], lane);
            // (normalised weights times columns, summed as columns: A1's columns are small behind the
            // front and large beside it, where weighted differences would lose digits)
            const Real w00 = p1 * p2 * W, w10 = g1 * p2 * lef.w, w01 = p1 * g2 * bel.w, w11 = g1 * g2 * bel_l.w;
            Col Nin = ColT<Real>::zero();
            if (act && l > 0) {
                const Real rn = Real(1) / ((w00 + w10) + (w01 + w11));
                Nin = ColT<Real>::fma_w(Nin, w00 * rn, N);
                Nin = ColT<Real>::fma_w(Nin, w01 * rn, mc_n(bel));
                Nin = ColT<Real>::fma_w(Nin, w10 * rn, mc_n(lef));
                Nin = ColT<Real>::fma_w(Nin, w11 * rn, mc_n(bel_l));
            }
            const Real nin = ColT<Real>::to_real(Nin);
            // the cell
            SrcRate<Real> r;
            CellODE<Real> C;
            C.ns = 1; C.c = alpha * n; C.r = &r; C.tabs = P.tabs;
            IntResult<Real> R;
            Real F0 = Real(0), dF0 = Real(0), f0 = Real(0);
            bool general = false;
            R.x = x0; R.IR = Real(0); R.lnfav = Real(0);
            r.A = r.b = r.Nin = r.p = Real(0);
            r.tab = tab;
            C.b0 = Real(1);
            if (act) {
                src_rate<Real>(r, qfac, tab, sig, dx, n, false, l, u, w, nin, P.tabs);
                C.b0 = tab < 0 ? r.b : sig * r.b;
                general = !integrate_prelude<Real, 1>(C, x0, dt, sig, R, F0, dF0, f0);
            }
            __syncwarp();
            a1_general<Real>(general, C, x0, dt, sig, F0, dF0, f0, R);
            Real dtau = -R.lnfav;
            if (!(dtau >= Real(0))) dtau = Real(0);
            N = act ? ColT<Real>::add(Nin, dtau / sig) : ColT<Real>::zero();
            W = act ? Real(1) / m_max(dtau, tau0) : Real(1);
            // a tied cell is written, and counted, by the lowest tied axis
            if (act && (axis == 0 || (u < l && (axis == 1 || w < l)))) {
                Nout[g] = nin;
                if (dt > Real(0)) {
                    xout[g] = R.x;
                    const double nV = double(n) * cellV;
                    ions += nV * double(x0 - R.x);
                    rec += nV * double(R.IR);
                }
            }
            const MCell<Real> own = mc_make(N, W);
            if (pub_r) mc_stcg(phalo + warp, own);
            if (warp < NW - 1) S.row[l & 1][warp][lane] = own;
            if (pub_a) mc_stcg(phalo + B + lane, own);
            march_sync<L::NC>();
        }
        if (tid == 0) mb_arrive(&S.done[b]);
    }
    // photon budget: one set of atomics per warp
    for (int o = 16; o > 0; o >>= 1) {
        ions += __shfl_down_sync(0xffffffffu, ions, o);
        rec += __shfl_down_sync(0xffffffffu, rec, o);
    }
    if (lane == 0 && (ions != 0.0 || rec != 0.0)) {
        DevState *st = G.st;
        atomicAdd(&st->bud_step[2], ions);
        atomicAdd(&st->bud_step[3], rec);
        atomicAdd(&st->bud_step[1], ions + rec);
    }
}

template <typename Real>
__global__ void __launch_bounds__(kMarchA1Warps * 32 + 32, 1) march_a1_kernel(MarchParams<Real> P)
{
    constexpr int NW = kMarchA1Warps;
    typedef MarchLayout<Real, NW, 1> L;
    __shared__ MarchShared<Real, NW, 1, kA1Chunk> S;
    const int tid = threadIdx.x;
    const unsigned epoch = march_begin(P, S);
    unsigned phase = 0;
    for (;;) {
        const unsigned tk = S.next;
        if (tk >= (unsigned)P.nitems) break;
        __syncthreads();
        const MarchItem it = P.items[tk];
        const March M = P.marches[it.march];
        const GridDev<Real> &G = P.grids[M.grid];
        const int c0 = it.l0 / kA1Chunk, c1 = (M.len - 1) / kA1Chunk;
        if (tid >= L::NC) march_hand<Real, NW, 1, kA1Chunk>(P, it, (int)tk, c0, c1, 0, M.len, epoch, phase, S);
        else march_a1_item<Real, NW>(P, it, M, G, c0, c1, phase, S);
        if (tid == L::NC) S.next = atomicAdd(P.ticket, 1u);
        __syncthreads();
        march_item_end(S, phase);
    }
    march_end(P, epoch);
}

template <typename Real> cudaError_t march_a1_occupancy(int *per_sm)
{
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, march_a1_kernel<Real>, kMarchA1Warps * 32 + 32, 0);
    if (e == cudaSuccess && *per_sm < 1) e = cudaErrorLaunchOutOfResources;
    return e;
}

template <typename Real>
cudaError_t launch_march_a1(const MarchParams<Real> &P, int nblocks, cudaStream_t s)
{
    if (P.nitems <= 0) return cudaSuccess;
    const int nb = nblocks < P.nitems ? (nblocks > 1 ? nblocks : 1) : P.nitems;
    march_a1_kernel<Real><<<nb, kMarchA1Warps * 32 + 32, 0, s>>>(P);
    return cudaGetLastError();
}

} // namespace oots
