// D2Q4 instantiations of the fused and the resident multi-update kernels (a
// translation unit of their own, to compile beside the lattice's others).
#include "mdf_res2d.cuh"

namespace mdf {

cudaError_t launch_fused_d2q4(int K, bool walls, const DevArgs &a, cudaStream_t s) {
  return K == 4 ? update_fused2d<D2Q4, 4>(walls, a, s)
       : K == 2 ? update_fused2d<D2Q4, 2>(walls, a, s) : cudaErrorInvalidValue;
}

cudaError_t launch_resident_d2q4(int steps, bool walls, const DevArgs &a, cudaStream_t s) {
  return update_resident2d<D2Q4>(walls, a, steps, s);
}
int resident_steps_d2q4(int nx, int ny, int nsets) {
  static OncePerDevice once;
  const ResShape r = res_shape(nx, ny, D2Q4::Q, nsets);
  return r.ctas && res_available(once, k_resident2d<D2Q4, true, FORCE_EQ321, true>) ? res_min_steps(r.rows * nx) : 0;
}

}  // namespace mdf
