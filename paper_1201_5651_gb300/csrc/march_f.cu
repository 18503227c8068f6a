// The column march instantiated for float (mixed path: float state, float-float columns).  One translation unit per
// precision so the two compile in parallel.
#include "march.cuh"

namespace oots {
template cudaError_t march_occupancy<float>(int, int *);
template cudaError_t launch_march<float>(const MarchParams<float> &, int, cudaStream_t);
template cudaError_t launch_pack_nx<float>(const GridDev<float> *, int, int, long long, int, cudaStream_t);
} // namespace oots
