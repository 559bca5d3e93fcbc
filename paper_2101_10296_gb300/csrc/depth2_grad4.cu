// Adjoint instantiations of the depth-2 kernel with 4 register qubits per
// thread.
#include "depth2_impl.cuh"

namespace qaoa {

template cudaError_t depth2_prepare_r<4, true>();
template const void *depth2_fn_r<4, true>(int);
template cudaError_t launch_depth2_r<4, true>(const RegLaunch &, int, cudaStream_t);

}  // namespace qaoa
