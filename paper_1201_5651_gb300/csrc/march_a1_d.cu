// The implicit scheme's march (A1) instantiated for double (FP64 path).  One translation
// unit per precision so the two compile in parallel.
#include "march_a1.cuh"

namespace oots {
template cudaError_t march_a1_occupancy<double>(int *);
template cudaError_t launch_march_a1<double>(const MarchParams<double> &, int, cudaStream_t);
} // namespace oots
