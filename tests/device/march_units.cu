// The march's reciprocal, square root and column sum, value by value, on the GPU.
// Test infrastructure: compiled by tests/test_gpu_march_units.py.
#include "../../paper_1201_5651_gb300/csrc/march.cuh"

using namespace oots;

__global__ void units_kernel(int m, const float *a, const float *b, float *rcp, float *root, float *hi, float *lo)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    rcp[i] = mr_rcp(a[i]);
    root[i] = mr_sqrt(a[i]);
    const ff s = col_step(ff{a[i], 0.0f}, b[i]);
    hi[i] = s.hi;
    lo[i] = s.lo;
}

extern "C" int oots_test_march_units(int m, const float *a, const float *b, float *out)
{
    units_kernel<<<(m + 255) / 256, 256>>>(m, a, b, out, out + m, out + 2 * (long long)m, out + 3 * (long long)m);
    return (int)cudaDeviceSynchronize();
}
