// Backprojector kernels of geometries whose LORs cross at most 4 slice(s) inside one pixel.
#include "backward.cuh"

namespace spdhg {
template cudaError_t launch_backward_nt<4>(const DevGeom&, int, int, const BwdArgs&, cudaStream_t);

}  // namespace spdhg
