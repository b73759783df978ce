// msh_staged_kt.cu -- the staged step (msh_staged.cuh) with the Kurganov-Tadmor flux, compiled apart in
// parallel with the other schemes.
#include "msh_staged.cuh"

namespace msh {
template cudaError_t launch_staged<float, 1>(const StagedArgs<float> &, int, cudaStream_t, int *);
template cudaError_t launch_staged<double, 1>(const StagedArgs<double> &, int, cudaStream_t, int *);
}  // namespace msh
