// msh_staged_hll.cu -- the staged step (msh_staged.cuh) with the HLL flux, compiled apart in
// parallel with the other schemes.
#include "msh_staged.cuh"

namespace msh {
template cudaError_t launch_staged<float, 0>(const StagedArgs<float> &, int, cudaStream_t, int *);
template cudaError_t launch_staged<double, 0>(const StagedArgs<double> &, int, cudaStream_t, int *);
}  // namespace msh
