// The allocation-free trace with its march left out: what the march would find in
// the counters it starts from.  Test infrastructure: compiled by
// tests/test_gpu_noalloc_counters.py.
#include "../../paper_1201_5651_gb300/csrc/common.cuh"
#include "../../paper_1201_5651_gb300/csrc/kernels.h"

static unsigned g_found[2];
namespace oots {
template <typename Real> static cudaError_t look(const MarchParams<Real> &P, cudaStream_t s)
{
    cudaError_t e = cudaMemcpyAsync(&g_found[0], P.ticket, sizeof(unsigned), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&g_found[1], P.done, sizeof(unsigned), cudaMemcpyDeviceToHost, s);
    return e == cudaSuccess ? cudaStreamSynchronize(s) : e;
}
template <> cudaError_t launch_march<float>(const MarchParams<float> &P, int, cudaStream_t s) { return look(P, s); }
template <> cudaError_t launch_march<double>(const MarchParams<double> &P, int, cudaStream_t s) { return look(P, s); }
template <> cudaError_t march_occupancy<float>(int, int *n) { *n = 1; return cudaSuccess; }
template <> cudaError_t march_occupancy<double>(int, int *n) { *n = 1; return cudaSuccess; }
} // namespace oots
#include "../../paper_1201_5651_gb300/csrc/noalloc.cu"

void oots_set_error_text(const char *) {}

// leaves both counters at `left`, calls the trace and returns what the march would have found (-1: error)
extern "C" long long oots_test_noalloc_counters(int precision, unsigned left, int n, const void *x, void *out)
{
    const unsigned v[2] = {left, left};
    if (cudaMemcpyToSymbol(g_noalloc_scratch, v, sizeof(v), kOffTicket) != cudaSuccess) return -1;
    const double pos[3] = {0.0, 0.0, 0.0};
    if (oots_trace_noalloc(0, precision, n, n, n, 1e16, nullptr, 100.0, x, pos, 6.3e-18, 0.6, out, nullptr, nullptr) != 0)
        return -1;
    return (long long)g_found[0] + g_found[1];
}
