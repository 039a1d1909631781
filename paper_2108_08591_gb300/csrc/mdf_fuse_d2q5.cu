// D2Q5 instantiations of the fused multi-update kernel (a translation unit of
// its own so that it compiles beside the lattice's other kernels).
#include "mdf_fuse2d.cuh"

namespace mdf {

cudaError_t launch_fused_d2q5(int K, bool walls, const DevArgs &a, cudaStream_t s) {
  return K == 4 ? update_fused2d<D2Q5, 4>(walls, a, s)
       : K == 2 ? update_fused2d<D2Q5, 2>(walls, a, s) : cudaErrorInvalidValue;
}

}  // namespace mdf
