// The implicit scheme's march (A1) instantiated for float (mixed path).  One translation
// unit per precision so the two compile in parallel.
#include "march_a1.cuh"

namespace oots {
template cudaError_t march_a1_occupancy<float>(int *);
template cudaError_t launch_march_a1<float>(const MarchParams<float> &, int, cudaStream_t);
} // namespace oots
