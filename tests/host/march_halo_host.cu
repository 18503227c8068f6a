// Host replay of the halo addresses of the column march (kernels.h: pyramids,
// blocks, published layers), as the handing warp stages them.  Test
// infrastructure: compiled by tests/test_march_halo_host.py.
#include "../../paper_1201_5651_gb300/csrc/common.cuh"
#include "../../paper_1201_5651_gb300/csrc/kernels.h"
#include <vector>

using namespace oots;

// Every cell that the blocks (32 x rows cells, chunks of H layers, aligned as
// the trace's when `sectors`) of one source at v stage from their neighbours:
// out[0] cells staged, out[1] of them outside the neighbour's published cells,
// out[2] layers before a marched one that the neighbour publishes and that are
// not staged.
extern "C" void oots_host_march_halo(int nx, int ny, int nz, const int *v, int rows, int H, int sectors, long long *out)
{
    out[0] = out[1] = out[2] = 0;
    for (int o = 0; o < 8; o++)
        for (int a = 0; a < 3; a++) {
            March M;
            if (!make_march(M, nx, ny, nz, v, o, a, nx, false)) continue;
            const int off = sectors ? M.off : 0, stride = rows + 32;
            const int n1 = march_nt1(M), n2 = march_nt2(M, rows);
            std::vector<MarchItem> items(n1 * n2);
            std::vector<long long> cells(n1 * n2);
            for (int t = 0; t < n1 * n2; t++) cells[t] = make_march_item(items[t], M, 0, t % n1, t / n1, rows);
            for (int t = 0; t < n1 * n2; t++) {
                const int T1 = t % n1, T2 = t / n1, l0 = items[t].l0;
                // the neighbour to the left, below and below left, and the cells of a layer staged from each
                const int up[3] = {T1 > 0 ? t - 1 : -1, T2 > 0 ? t - n1 : -1, T1 > 0 && T2 > 0 ? t - n1 - 1 : -1};
                const int lo[3] = {0, rows, rows - 1}, hi[3] = {rows, stride, rows};
                for (int k = 0; k < 3; k++) {
                    if (up[k] < 0) continue;
                    const int first = items[up[k]].l0;
                    std::vector<bool> have(M.len, false);
                    for (int c = (l0 + off) / H; c <= (M.len - 1 + off) / H; c++)
                        for (int s = 0; s < H; s++) {
                            const int l = c * H - off - 1 + s;
                            if (!march_published(l, first, M.len)) continue;
                            if (l >= 0 && l < M.len) have[l] = true;
                            for (int e = lo[k]; e < hi[k]; e++) {
                                const long long at = (long long)(l - first) * stride + e;
                                out[0]++;
                                out[1] += at < 0 || at >= cells[up[k]];
                            }
                        }
                    for (int l = l0 > 0 ? l0 - 1 : 0; l + 1 < M.len; l++) out[2] += l >= first && !have[l];
                }
            }
        }
}

// the computing warps' limit on their wait for the halo (kernels.h)
extern "C" long long oots_host_march_ready_limit(long long spin_limit) { return march_ready_limit(spin_limit); }
