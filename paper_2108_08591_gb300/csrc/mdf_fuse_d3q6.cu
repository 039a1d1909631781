// D3Q6 instantiations of the fused two-update kernel (a translation unit of its
// own so that it compiles beside the lattice's other kernels).
#include "mdf_fuse3d.cuh"

namespace mdf {

cudaError_t launch_fused_d3q6(int K, bool walls, const DevArgs &a, cudaStream_t s) {
  return K == 2 ? update_fused3d<D3Q6>(walls, a, s) : cudaErrorInvalidValue;
}

}  // namespace mdf
