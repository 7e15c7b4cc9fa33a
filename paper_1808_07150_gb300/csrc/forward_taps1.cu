// Forward projector kernels of geometries whose LORs cross at most 1 slice(s) inside one pixel.
#include "forward.cuh"

namespace spdhg {
template cudaError_t launch_forward_nt<1>(const DevGeom&, int, int, const FwdArgs&, cudaStream_t);
}  // namespace spdhg
