// Adjoint instantiations of the depth-2 kernel with 5 register qubits per
// thread.
#include "depth2_impl.cuh"

namespace qaoa {

template cudaError_t depth2_prepare_r<5, true>();
template const void *depth2_fn_r<5, true>(int);
template cudaError_t launch_depth2_r<5, true>(const RegLaunch &, int, cudaStream_t);

}  // namespace qaoa
