// The implicit wavefront sweep (A1) instantiated for double (FP64 path).  One translation
// unit per precision so the two compile in parallel.
#include "sweep_impl.cuh"

namespace oots {
template bool sweep_shape_ok<double>(int);
template int sweep_occupancy<double>(int);
template cudaError_t prepare_sweeps<double>();
template cudaError_t launch_sweep<double>(const SweepParams<double> &, int, int, cudaStream_t);
} // namespace oots
