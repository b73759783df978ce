// msh_staged_roe.cu -- the staged step (msh_staged.cuh) with the Roe-type flux, compiled apart in
// parallel with the other schemes.
#include "msh_staged.cuh"

namespace msh {
template cudaError_t launch_staged<float, 3>(const StagedArgs<float> &, int, cudaStream_t, int *);
template cudaError_t launch_staged<double, 3>(const StagedArgs<double> &, int, cudaStream_t, int *);
}  // namespace msh
