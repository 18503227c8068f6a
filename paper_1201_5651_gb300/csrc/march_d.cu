// The column march instantiated for double (FP64 path).  One translation unit per
// precision so the two compile in parallel.
#include "march.cuh"

namespace oots {
template cudaError_t march_occupancy<double>(int, int *);
template cudaError_t launch_march<double>(const MarchParams<double> &, int, cudaStream_t);
template cudaError_t launch_pack_nx<double>(const GridDev<double> *, int, int, long long, int, cudaStream_t);
} // namespace oots
