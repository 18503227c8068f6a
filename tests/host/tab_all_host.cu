// Host build of the shared table read (tab_all) beside the three functions it
// stands for.  Test infrastructure: compiled by tests/test_tab_all_host.py.
#include "integrator_host.cu"

template <typename Real> static void tab_both(const DevTable<Real> &T, const double *N, const double *dN, int m, double *out)
{
    for (int i = 0; i < m; i++) {
        const Real a = Real(N[i]), b = Real(dN[i]);
        Real lnp, dl, slope;
        tab_all(T, a, b, lnp, dl, slope);
        const double v[6] = {double(lnp), double(dl), double(slope), double(tab_lnp(T, a)), double(tab_dlnp(T, a, b)),
                             double(tab_dlnp_dN(T, a + b))};
        for (int q = 0; q < 6; q++) out[6 * i + q] = v[q];
    }
}

// the table's node columns; returns how many
extern "C" int oots_host_tab_nodes(double Tbb, double sigma0, double *out)
{
    const HostTable &H = host_table(1, Tbb, sigma0);
    HostDevTable<double> D(H);
    for (int k = 0; k < D.T.K; k++) out[k] = D.T.Nnode[k];
    return D.T.K;
}

extern "C" void oots_host_tab_both(int precision, double Tbb, double sigma0, const double *N, const double *dN, int m,
                                   double *out)
{
    const HostTable &H = host_table(1, Tbb, sigma0);
    if (precision == 0) {
        HostDevTable<double> D(H);
        tab_both(D.T, N, dN, m, out);
    } else {
        HostDevTable<float> D(H);
        tab_both(D.T, N, dN, m, out);
    }
}
